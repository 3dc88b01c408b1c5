// build.cu -- stage 2 of the GraceKV pass: one prototype tree per
// layer-KV-head-slot unit (App. A.2 atomic units), built level by level by one
// CTA that keeps the whole slot in shared memory.
//
// Per unit (l, g, j), slot [sa, sb), n <= 128 tokens:
//   E[t][u] = exp(q_u . k_t / sqrt d - m_u)   distortion probe u uses query
//             head H(g)[u mod |H(g)|] (App. A.3, GQA round robin), m_u its
//             max logit over [0, T)
//   k_circ_t = RoPE^-1(k_t, t)                 (Eq. app_rope_prototype)
// For every node I = [a, b) of a level, the candidate children are prefixes
// [a, xi) and suffixes [xi, b) of I for the binary cuts X_v (top-16 positions
// by curvature in [a, b-2], cut xi = t + 1, plus the midpoint; App. B.4
// Eq. app_tree_split_candidates) and the two sides of the salient-token
// extraction at p* = argmax R_tok (Eq. app_extract_split).  The sides of the
// cut of largest curvature reward are evaluated first; cuts and extractions
// that an exact bound then rules out are never evaluated (phase D1).  For each
// evaluated candidate J the prototype (ktil, vtil, m_eff; Eqs. app_rope_prototype,
// app_value_prototype, app_effective_multiplicity) is formed by direct sums
// over J; then a forward scan (prefixes) and a backward scan (suffixes) over
// the node's tokens accumulate Z_u(J) and M_u(J) (Eq.
// app_original_attention_stats) for every probe and evaluate D_u (Eq.
// app_probe_distortion) at each candidate end, weighted by the attention mass
// Z_u(J) / Z_u (Eq. app_node_and_drop_distortion).  The refinement form
// follows Eqs. app_binary_split .. app_split_choice; gains, costs and
// utilities follow Eqs. app_operation_gains .. app_unit_utility (clamped at
// 0); each Split op also gets its bottleneck key kappa = min(U, kappa of the
// op that created the node), which the allocator's threshold select uses.
//
// Pruned construction.  A launch evaluates at most `max_levels` levels; the
// nodes below stay pending (child count -1, no Split op yet) and each unit
// reports the largest key of the ops that created its pending nodes.  The
// host then computes the allocation threshold tau over the ops built so far
// -- tau can only grow as ops are added, so it never exceeds the final
// threshold -- and resumes only the pending nodes whose creator has a key
// >= tau: a node whose creator's key is below the final threshold never
// reaches the frontier before the allocation stops, so its own Split is never
// needed.  Resuming repeats until no pending node qualifies.  Within a launch
// a child whose bound is below the launch's tau stays pending as well, so a
// resume launch may build several levels without expanding what its tau
// already rules out.
//
// Layout.  256 threads per scan direction; thread (p, c) owns the probes p and p + 32 and the
// elements 4 c + 32 g + j (j < 4) of every d-vector: each value, prototype or
// key chunk it reads from shared memory serves two probes, and 8 consecutive
// threads read 128 contiguous bytes (one wavefront, no bank conflicts).
// Three instances by slot length: up to 36 tokens three CTAs fit on an SM, up to
// 64 two; up to 128 tokens one CTA of 512 threads scans both directions at once.
#include "gkv_internal.cuh"

#include <cfloat>

#include <type_traits>

namespace gkv {
namespace {

constexpr int kMaxCuts = 18;     // K + midpoint, K <= 16 (+1 spare)
constexpr int kNT = 256;         // threads of one scan direction (a CTA has one or two, Smem::DIRS)
constexpr int kNPP = 32;         // probe pairs: thread handles probes p and p + 32 (W <= 64)
constexpr int kNCL = 8;          // threads per probe pair (4-element groups, interleaved)
constexpr int kPPW = 32 / kNCL;  // probe pairs per warp: lane = 4 c + (pair % 4), so that the
                                 // 4 lanes reading one 16-byte chunk are adjacent (one shared-
                                 // memory wavefront serves them; lanes 8 apart would not merge)
// A cut evaluated ahead of the others pays where its reward rules most of them
// out, and costs a second sweep of the node where it does not: with
// lambda_kappa at most kDirect of the node's D (of a fresh root's attention mass,
// which weights its D, not known yet) all cuts are evaluated at once.  The mass
// is formed below kDirectMax only: a slot of a long request holds far less.
// 16 layers of llama32k, lambda_kappa 0 at 8x / 32x: 100.2 -> 81.9 / 35.0 ->
// 29.2 ms, 2e-4: 95.4 -> 83.0 / 34.5 -> 29.7, 1e-3: 75.2 -> 67.9 / 29.6 -> 27.4;
// shares of 0.1 to 0.5 were up to 5 % slower at 1e-4 to 1e-3, of 2 and 3 no faster.
constexpr float kDirect = 1.0f, kDirectRoot = 1.0f, kDirectMax = 0.01f;
constexpr int kNCR = 19;         // candidate rows held at a time: 17 cuts + p* side (+ 1)

struct BuildArgs {
    const void *K, *V, *Q;
    const int32_t *slots;
    const float2 *rope;
    const double *kappa;
    const float *rtok, *row_m, *row_Z, *omega;
    const float *Eg;             // nullable: [L G][N_c][32][2] probe weights of every token (score pass B)
    const uint8_t *fl_acc;       // nullable: [L G][N_c] accepted singleton-floor positions
    const float *fl_f;           //           and their floor scores
    int L, G, Hq, T, d, W, gq, cs, Nc, J, k_cand;
    float inv_sqrt_d, lamZ, lamM, eps;
    float lam_kappa, base_frac;
    int prune;                   // lambda_Z, lambda_M >= 0, so every D >= 0: cuts and nodes may be ruled out by bounds
    // work list: fresh launches index (slot list entry, lg), resume launches units
    int resume;                  // 0: build from the root, 1: resume pending nodes
    int root_only;               // fresh: evaluate only the root's own distortion (split stays pending)
    int max_levels;              // levels evaluated by this launch
    int nrow;                    // candidate rows that the launch's shared memory holds (kNCR or Smem::NROW)
    float tau;                   // resume: evaluate pending nodes whose key bound >= tau
    const int32_t *list;         // fresh: slot indices; resume: unit ids; subtree: node indices
    int64_t stride;              // the launch's classes follow one another at this distance,
    int c1, c2;                  // its work items c1.. and c2.. in the second and third
    int lg0, nlg;                // fresh: the (l, g) range [lg0, lg0 + nlg) of the launch
    // outputs
    int32_t *nd_a, *nd_b, *nd_child0, *nd_parent, *nd_unit;
    int8_t *nd_nchild, *nd_cost;
    float *nd_D;
    float *nd_R, *nd_U, *nd_kappa;
    uint8_t *nd_sel;
    uint2 *ops;                  // compact list of the Split ops (allocation input)
    unsigned int *n_ops;
    int32_t *u_nnodes;
    float *u_Uadd, *u_Ddrop, *u_pend;
    uint8_t *u_sel;
    int *status;
    unsigned long long *work;
};

struct NodeS {
    float D;
    float kin;                   // bottleneck key of the op that created the node
    short a, b;
    signed char nchild;          // -1: pending (not evaluated)
};

struct BatchNode {
    unsigned long long klo, khi;   // smallest and largest curvature key over the node's cut positions
    float kh[kMaxCuts];      // normalised curvature of the cuts
    float cD[3];
    unsigned more, keep;     // open node: cuts that the first one evaluated does not rule out; nor their D_L
    short node, pstar;
    short op;                // the node's place among the batch's Split ops (-1: none)
    short ca[3], cb[3];
    int8_t cut[kMaxCuts];    // local cut positions xi (ascending)
    int8_t ncut, k1;         // cuts; the one of largest curvature reward
    int8_t rl, rr, whole;    // rows of its sides (-1: single token) and of the node itself
    int8_t direct;           // no cut is evaluated ahead of the others
    int8_t np, ns;           // open node: prefixes and suffixes left to evaluate
    int8_t nchild;           // -1: pending root, -2: undecided
    int8_t forced;           // extraction at a singleton-floor position (a floor op)
    int8_t ext;              // the extraction's sides are needed
    int8_t pre_b, pre_e, suf_b, suf_e;   // rows: prefixes (ascending end), suffixes (descending start)
};

struct Cand {
    short a, b;      // local interval (a == b: unused entry)
    float meff;
};

// Sums of two products round one product and fuse the other.  Which one is
// written out, so that the compiler's choice cannot move a result's last bit
// (and with it a near-tie between cuts) from one build or instance to another.
__device__ __forceinline__ void rotate_back(float x, float y, float c, float s, float &lo, float &hi) {
    lo = fmaf(x, c, y * s);
    hi = fmaf(y, c, -(x * s));
}
template <bool SINE_FUSED>
__device__ __forceinline__ void rotate_to(float x, float y, float c, float s, float &lo, float &hi) {
    lo = fmaf(x, c, -(y * s));
    hi = SINE_FUSED ? fmaf(x, s, y * c) : fmaf(y, c, x * s);
}

// Upper bound of a split's utility: U = omega R (D - sum D_children) / cost
// <= omega R D where every D and omega are >= 0, since cost >= 1 (Eqs.
// app_operation_gains, app_unit_utility).  Rounded up by 1e-5 of its value: the R that the bound
// uses (one fp32 sum over the node's tokens) and the R of the later gain (the
// sum of its children's sums) differ by at most ~1.3e-6 of R, and the products
// add a few ulp, so rounding never makes a bound fall below the utility it bounds.
__device__ __forceinline__ float key_bound(float x) {
    return x + fabsf(x) * 1e-5f;
}

// Order-preserving 64-bit key of a double (larger value -> larger key), so
// that curvature ranks compare exactly like the fp64 values with integer ops.
__device__ __forceinline__ unsigned long long okey(double x) {
    unsigned long long u = (unsigned long long)__double_as_longlong(x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double okey_inv(unsigned long long k) {
    unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)u);
}

// 8 consecutive input elements held raw in registers (the load is issued
// first, the conversion to fp32 happens at get).
template <typename T> struct Raw8;
template <> struct Raw8<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float *p) {
        a = reinterpret_cast<const float4 *>(p)[0];
        b = reinterpret_cast<const float4 *>(p)[1];
    }
    __device__ __forceinline__ void get(float v[8]) const {
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
};
template <> struct Raw8<__nv_bfloat16> {
    uint4 u;
    __device__ __forceinline__ void load(const __nv_bfloat16 *p) { u = *reinterpret_cast<const uint4 *>(p); }
    __device__ __forceinline__ void get(float v[8]) const {
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {   // bf16 -> fp32 is exact: the bits move to the high half
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
};

__device__ __forceinline__ int round_half_even_mid(int a, int b) {
    int s = a + b - 1;
    if ((s & 1) == 0) return s >> 1;
    int lo = (s - 1) >> 1;
    return (lo & 1) == 0 ? lo : lo + 1;
}

// 4 consecutive elements (8- or 16-byte aligned) as floats.
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16 *p) {
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}

// Row that a lane of an 8-row matrix tile reads in an instance of NMAX rows:
// where they are no multiple of 8, the slot's last one in place of those past
// it (the columns of rows past the slot are dropped).
template <int NMAX>
__host__ __device__ constexpr int tile_row(int row, int n) { return NMAX % 8 == 0 || row < n ? row : n - 1; }
template <int NMAX>
constexpr bool tile_rows_inside() {
    for (int n = 1; n <= NMAX; n++)
        for (int row = 0; row < (n + 7) / 8 * 8; row++)
            if (tile_row<NMAX>(row, n) >= NMAX) return false;
    return true;
}
static_assert(tile_rows_inside<kTinyUnit>() && tile_rows_inside<kShortUnit>() && tile_rows_inside<kMaxUnit>(),
              "the probe weights' tiles stay inside the slot's array");

// 8 floats to a 16-byte aligned shared-memory row.
__device__ __forceinline__ void st8(float *p, const float v[8]) {
    reinterpret_cast<float4 *>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4 *>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
}

// Order-preserving 32-bit key of a float (-0 and +0 alike).
__device__ __forceinline__ unsigned fkey_ordered(float x) {
    const unsigned u = __float_as_uint(x + 0.f);
    return u >> 31 ? ~u : u | 0x80000000u;
}

// Sum over a probe pair's 8 chunk lanes (lane bits 2..4) of each of 8 values,
// as a reduce-scatter: 7 exchanges instead of the 24 of 8 butterflies, and the
// lane with chunk index c ends with the sum of v[c].  Every sum pairs the
// lanes in the butterfly's order (bit 2, then 3, then 4), so its bits are the
// butterfly's.
__device__ __forceinline__ float reduce_scatter8(const float v[8], int lane) {
    float x[4], y[2];
    const bool h0 = lane & kPPW, h1 = lane & (2 * kPPW), h2 = lane & (4 * kPPW);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const float send = h0 ? v[2 * i] : v[2 * i + 1], keep = h0 ? v[2 * i + 1] : v[2 * i];
        x[i] = keep + __shfl_xor_sync(0xffffffffu, send, kPPW);
    }
#pragma unroll
    for (int i = 0; i < 2; i++) {
        const float send = h1 ? x[2 * i] : x[2 * i + 1], keep = h1 ? x[2 * i + 1] : x[2 * i];
        y[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * kPPW);
    }
    const float send = h2 ? y[0] : y[1], keep = h2 ? y[1] : y[0];
    return keep + __shfl_xor_sync(0xffffffffu, send, 4 * kPPW);
}

// The same over four values; lane c ends with the sum of v[c & 3] (both halves
// of the lanes hold it).
__device__ __forceinline__ float reduce_scatter4(float v0, float v1, float v2, float v3, int lane) {
    const bool h0 = lane & kPPW, h1 = lane & (2 * kPPW);
    const float x0 = (h0 ? v1 : v0) + __shfl_xor_sync(0xffffffffu, h0 ? v0 : v1, kPPW);
    const float x1 = (h0 ? v3 : v2) + __shfl_xor_sync(0xffffffffu, h0 ? v2 : v3, kPPW);
    const float y = (h1 ? x1 : x0) + __shfl_xor_sync(0xffffffffu, h1 ? x0 : x1, 2 * kPPW);
    return y + __shfl_xor_sync(0xffffffffu, y, 4 * kPPW);
}

// Running sums of an interval's prototype: PPL rotation pairs (i, i + d/2) per
// lane, PPL consecutive i (a packed pair when PPL = 2; each lane of a packed
// add or FMA rounds like the scalar one).
template <int PPL, int HALF> struct KeySum;     // sum k_circ of both halves, sum ||k||
template <int HALF> struct KeySum<2, HALF> {
    float2 m0, m1;
    float ks;
    __device__ __forceinline__ void clear() { m0 = m1 = make_float2(0.f, 0.f); ks = 0.f; }
    __device__ __forceinline__ void add(const float *k, float kn) {
        m0 = fadd2(m0, *reinterpret_cast<const float2 *>(k));
        m1 = fadd2(m1, *reinterpret_cast<const float2 *>(k + HALF));
        ks += kn;
    }
    __device__ __forceinline__ float lo(int j) const { return j ? m0.y : m0.x; }
    __device__ __forceinline__ float hi(int j) const { return j ? m1.y : m1.x; }
};
template <int HALF> struct KeySum<1, HALF> {
    float m0, m1, ks;
    __device__ __forceinline__ void clear() { m0 = m1 = ks = 0.f; }
    __device__ __forceinline__ void add(const float *k, float kn) {
        m0 += k[0];
        m1 += k[HALF];
        ks += kn;
    }
    __device__ __forceinline__ float lo(int) const { return m0; }
    __device__ __forceinline__ float hi(int) const { return m1; }
};
template <int PPL, int HALF> struct ValueSum;   // sum R v and sum v of both halves, sum R
template <int HALF> struct ValueSum<2, HALF> {
    float2 r0, r1, s0, s1;
    float rs;
    __device__ __forceinline__ void clear() { r0 = r1 = s0 = s1 = make_float2(0.f, 0.f); rs = 0.f; }
    __device__ __forceinline__ void add(const float *v, float r) {
        const float2 x0 = *reinterpret_cast<const float2 *>(v), x1 = *reinterpret_cast<const float2 *>(v + HALF);
        const float2 rr = make_float2(r, r);
        r0 = ffma2(rr, x0, r0);
        r1 = ffma2(rr, x1, r1);
        s0 = fadd2(s0, x0);
        s1 = fadd2(s1, x1);
        rs += r;
    }
    __device__ __forceinline__ float rlo(int j) const { return j ? r0.y : r0.x; }
    __device__ __forceinline__ float rhi(int j) const { return j ? r1.y : r1.x; }
    __device__ __forceinline__ float slo(int j) const { return j ? s0.y : s0.x; }
    __device__ __forceinline__ float shi(int j) const { return j ? s1.y : s1.x; }
};
template <int HALF> struct ValueSum<1, HALF> {
    float r0, r1, s0, s1, rs;
    __device__ __forceinline__ void clear() { r0 = r1 = s0 = s1 = rs = 0.f; }
    __device__ __forceinline__ void add(const float *v, float r) {
        r0 = fmaf(r, v[0], r0);
        r1 = fmaf(r, v[HALF], r1);
        s0 += v[0];
        s1 += v[HALF];
        rs += r;
    }
    __device__ __forceinline__ float rlo(int) const { return r0; }
    __device__ __forceinline__ float rhi(int) const { return r1; }
    __device__ __forceinline__ float slo(int) const { return s0; }
    __device__ __forceinline__ float shi(int) const { return s1; }
};

// A node's decision: extraction at its p* (Eq. app_extract_split).
__device__ __forceinline__ void set_extraction(BatchNode &B, int a, int b, float DL, float DR) {
    const int ps = B.pstar;
    int ne = 0;
    if (ps > a) { B.ca[ne] = (short)a; B.cb[ne] = (short)ps; B.cD[ne] = ps - a >= 2 ? DL : 0.f; ne++; }
    B.ca[ne] = (short)ps; B.cb[ne] = (short)(ps + 1); B.cD[ne] = 0.f; ne++;
    if (ps + 1 < b) { B.ca[ne] = (short)(ps + 1); B.cb[ne] = (short)b; B.cD[ne] = b - ps - 1 >= 2 ? DR : 0.f; ne++; }
    B.nchild = (int8_t)ne;
}

// Instances by slot length: up to kTinyUnit tokens three CTAs per SM, up to
// kShortUnit two, longer slots one CTA of twice the threads.
template <int DH, int NMAX>
struct Smem {
    static constexpr int DIRS = NMAX <= kShortUnit ? 1 : 2;   // scan directions that run side by side
    static constexpr int CTAS = NMAX <= kTinyUnit ? 3 : (NMAX <= kShortUnit ? 2 : 1);   // per SM
    static constexpr int NT = kNT * DIRS;
    static constexpr int NWARPS = NT / 32;
    static constexpr int NB = NWARPS;        // nodes per batch: one a warp
    static constexpr int MAXNODES = 2 * NMAX;
    static constexpr int NROW = kNCR * DIRS; // candidate rows held at a time: one side of a node, or both
    static constexpr int KTW = DH < 128 ? 128 : DH;        // a row also holds 32 float4 of sums
    static constexpr int MW = (MAXNODES + 31) / 32;
    static constexpr int KPAD = NMAX <= kShortUnit ? 8 : 0;
    float kc[NMAX][DH + KPAD];               // rows padded by 32 B where there is room: the probe-weight
                                             // MMA reads 8 rows at once, which then fall in distinct banks
    float vv[NMAX][DH];                      // values, converted once to fp32
    float2 E[NMAX][kNPP];                    // probe weights of probes (p, p + 32)
    float2 RK[NMAX];                         // token value, ||k||
    unsigned long long kap[NMAX];            // order-preserving keys of the curvature
    uint8_t rk[NMAX];                        // the token's place among the slot's by curvature (0: largest)
    BatchNode bn[NB];
    Cand cand[NROW];
    NodeS nodes[MAXNODES];
    float Ff[NMAX];                          // floor score of an accepted floor position, -inf elsewhere
    float candD[NROW + kNCR], candP[NROW + kNCR];  // per-row D and drop mass (prefixes kept while the suffixes follow)
    unsigned lvl[2][MW];                     // nodes of the level (bit masks), of the next one
    unsigned op_base;                        // the batch's first Split op in the global list
    unsigned int wcnt[NWARPS][3];            // per-warp work counters
    float pend;
    float rootR;                             // R of a fresh root
    // Candidate rows, each: the key prototype (KTW; once the logits are taken,
    // (residual / ||M||^2, Z) of the probes p and p + 32), the value prototype (DH)
    // and m_eff exp(logit) of the probes (p, p + 32).  The 128-token instance keeps
    // a row together, so that its last rows may lie past the launch's shared memory
    // (A.nrow); the others keep the parts apart (1 % faster).
    static constexpr int ROWF = KTW + DH + 2 * kNPP;
    alignas(16) float rows[NROW * ROWF];
    __device__ __forceinline__ float *ktil(int r) { return rows + r * (DIRS == 2 ? ROWF : KTW); }
    __device__ __forceinline__ float *vtil(int r) { return rows + (DIRS == 2 ? r * ROWF + KTW : NROW * KTW + r * DH); }
    __device__ __forceinline__ float2 *zt(int r) {
        return reinterpret_cast<float2 *>(rows + (DIRS == 2 ? r * ROWF + KTW + DH : NROW * (KTW + DH) + r * 2 * kNPP));
    }
};

// SUB: the subtree mode, a compile-time flag so that the other instances carry
// none of its index mapping: the list holds pending nodes of at most NMAX
// tokens inside long units (build_long.cu), as global node indices; each CTA
// builds its node's subtree to the leaves into the node slots reserved for it
// (the unit-relative index in its child0)
template <int DH, typename Tin, int NMAX, bool SUB>
__global__ void __launch_bounds__(Smem<DH, NMAX>::NT, Smem<DH, NMAX>::CTAS) unit_build_kernel(BuildArgs A) {
    using S = Smem<DH, NMAX>;
    // thread (p, c): probes p and p + 32, elements 4 c + 32 g + j (g < NG, j < 4)
    constexpr int HALF = DH / 2, NWARPS = S::NWARPS, NG = DH / (4 * kNCL), CH = 4 * NG;
    constexpr int NT = S::NT, DIRS = S::DIRS;
    static_assert(kNPP * kNCL == kNT && DH % (4 * kNCL) == 0, "probe layout");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S &sm = *reinterpret_cast<S *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int dwarp = warp & (kNT / 32 - 1);   // warp within its scan direction (DIRS = 2: warps 8..15 take the suffixes)
    int j, lg;
    auto item = [&](int i) {
        const int q = (i >= A.c1) + (i >= A.c2);
        return A.list[q * A.stride + i - (q == 0 ? 0 : (q == 1 ? A.c1 : A.c2))];
    };
    int64_t gv_sub = -1;         // subtree mode: the pending node whose subtree this CTA builds
    if constexpr (SUB) {
        gv_sub = item(blockIdx.x);
        const int uidr = A.nd_unit[gv_sub];
        lg = uidr / A.J;
        j = uidr - lg * A.J;
    } else if (A.resume) {
        const int uidr = item(blockIdx.x);
        lg = uidr / A.J;
        j = uidr - lg * A.J;
    } else {
        j = item(blockIdx.x / A.nlg);   // slot-major: the units of a slot share its table rows
        lg = A.lg0 + blockIdx.x % A.nlg;
    }
    const bool fresh = !A.resume && !SUB;
    const int l = lg / A.G, g = lg - l * A.G;
    const int64_t uid = (int64_t)lg * A.J + j;
    const int64_t nbase = node_base(lg, A.slots[j], A.cs, A.Nc);   // the unit's node slots
    // the tokens held: the slot, or in subtree mode the node's interval
    const int sa = SUB ? A.nd_a[gv_sub] : A.slots[j];
    const int sb = SUB ? A.nd_b[gv_sub] : A.slots[j + 1];
    const int n = sb - sa;
    // global node index of local node k, and its index inside the unit: the
    // local nodes of a subtree are its root and then its reserved slots
    const int64_t sub_res = SUB ? (int64_t)A.nd_child0[gv_sub] : 0;
    auto gidx = [&](int k) -> int64_t {
        if constexpr (SUB) return k == 0 ? gv_sub : nbase + sub_res + (k - 1);
        else return nbase + k;
    };
    if (n < 1 || n > NMAX) {
        if (tid == 0) atomicOr(A.status, 4);
        return;
    }
    const Tin *Kp = static_cast<const Tin *>(A.K) + ((size_t)lg * A.T + sa) * DH;
    const Tin *Vp = static_cast<const Tin *>(A.V) + ((size_t)lg * A.T + sa) * DH;
    const float om = A.omega ? A.omega[lg] : 1.0f;
    // key bound of a pending node of value R and distortion D, kin the key of its
    // creator; with a negative weight or omega only the creator's key bounds it
    const bool bounded = A.prune && om >= 0.f;
    auto split_bound = [&](float kin, float R, float D) { return bounded ? fminf(kin, key_bound(om * R * D)) : kin; };

    // Probe weights E[t][u] (Eq. app_probe_distortion), stored at E[t][u % 32].x
    // (u < 32) or .y (u >= 32).  When the score pass wrote them for every token
    // they are copied in with the slot (cp.async, 16 bytes each); otherwise
    // they are formed below from the raw keys.
    float *Ef = reinterpret_cast<float *>(&sm.E[0][0]);
    auto eidx = [](int t, int u) { return t * 2 * kNPP + 2 * (u & (kNPP - 1)) + (u >> 5); };
    if (A.Eg) {   // the same layout, n rows of 256 bytes: 16-byte copies
        const float *Eu = A.Eg + ((size_t)lg * A.Nc + (sa - A.cs)) * (2 * kNPP);
        for (int idx = tid; idx < n * (2 * kNPP / 4); idx += NT) cp_async16(Ef + 4 * idx, Eu + 4 * idx, true);
        cp_async_commit();
    }
    // resume: the unit's node records, one per thread (a unit has at most
    // 2 n - 1 <= NT of them), loaded beside the slot
    int nn = 0;
    int32_t rec_a = 0, rec_b = 0, rec_p = -1;
    int rec_nch = 0;
    float rec_D = 0.f, rec_U = 0.f, rec_kin = 0.f;
    const bool resume = !SUB && A.resume;
    if (resume) {
        nn = A.u_nnodes[uid];
        if (tid < nn) {
            const int64_t v = nbase + tid;
            rec_a = A.nd_a[v]; rec_b = A.nd_b[v]; rec_p = A.nd_parent[v];
            rec_nch = A.nd_nchild[v];
            rec_D = A.nd_D[v]; rec_U = A.nd_U[v];
        }
    }
    // ---- load the slot ------------------------------------------------------
    const bool own = tid < n;   // n <= NT
    const double kapv = own ? A.kappa[sa + tid] : 0.0;
    const float rtv = own ? A.rtok[(size_t)lg * A.Nc + (sa - A.cs) + tid] : 0.f;
    bool bad = own && !isfinite(rtv);   // non-finite probe weights or token values
    bool rotated = false;
    if constexpr (std::is_same<Tin, __nv_bfloat16>::value) {
        if (A.Eg) {
            // Only the rotated keys are needed: HALF / 8 consecutive threads
            // hold a token, each the 8 rotation pairs (i, i + d/2) from its
            // i; keys, values and rotations are all loaded before any is used.
            // The thread also forms its part of ||k_t||^2, which equals
            // ||k_circ_t||^2 (a rotation keeps the norm).
            rotated = true;
            constexpr int TPT = HALF / 8, TPI = NT / TPT;   // threads per token, tokens per iteration
            const int i = (tid % TPT) * 8;
            for (int t0 = 0; t0 < n; t0 += TPI) {
                const int t = t0 + tid / TPT;
                const bool in = t < n;
                Raw8<Tin> k0, k1, v0, v1;
                float4 cs[4];
                if (in) {
                    const size_t e = (size_t)t * DH + i;
                    k0.load(Kp + e); k1.load(Kp + e + HALF);
                    v0.load(Vp + e); v1.load(Vp + e + HALF);
                    const float4 *rp = reinterpret_cast<const float4 *>(A.rope + (size_t)(sa + t) * HALF + i);
#pragma unroll
                    for (int q = 0; q < 4; q++) cs[q] = rp[q];
                }
                float ss0 = 0.f, ss1 = 0.f;
                if (in) {
                    float x[8], y[8], lo[8], hi[8];
                    k0.get(x);
                    k1.get(y);
#pragma unroll
                    for (int u = 0; u < 8; u++) {
                        const float cx = u & 1 ? cs[u / 2].z : cs[u / 2].x, cy = u & 1 ? cs[u / 2].w : cs[u / 2].y;
                        ss0 = fmaf(x[u], x[u], ss0);
                        ss1 = fmaf(y[u], y[u], ss1);
                        rotate_back(x[u], y[u], cx, cy, lo[u], hi[u]);
                    }
                    st8(&sm.kc[t][i], lo);
                    st8(&sm.kc[t][i + HALF], hi);
                    v0.get(x);
                    v1.get(y);
                    st8(&sm.vv[t][i], x);
                    st8(&sm.vv[t][i + HALF], y);
                }
#pragma unroll
                for (int o = 1; o < TPT; o <<= 1) {   // the chunks of each half, then the halves
                    ss0 += __shfl_xor_sync(0xffffffffu, ss0, o);
                    ss1 += __shfl_xor_sync(0xffffffffu, ss1, o);
                }
                if (in && i == 0) sm.RK[t].y = sqrtf(ss0 + ss1);
            }
        }
    }
    if (!rotated) {
        // DH / 8 consecutive threads hold a token; every load of a group is
        // issued before any is used
        constexpr int TPT = DH / 8, GRP = 2;
        const int iters = (n * DH + NT * 8 - 1) / (NT * 8);
        for (int i0 = 0; i0 < iters; i0 += GRP) {   // the same trip counts for every thread
            Raw8<Tin> kr[GRP], vr[GRP];
#pragma unroll
            for (int q = 0; q < GRP; q++) {
                const int e = (i0 + q) * NT * 8 + tid * 8;
                if (i0 + q < iters && e < n * DH) {
                    kr[q].load(Kp + e);
                    vr[q].load(Vp + e);
                }
            }
#pragma unroll
            for (int q = 0; q < GRP; q++) {
                if (i0 + q >= iters) break;
                const int e = (i0 + q) * NT * 8 + tid * 8;
                const bool in = e < n * DH;
                const int t = e / DH, i = e - t * DH;
                float ss = 0.f;
                if (in) {
                    float kx[8], vx[8];
                    kr[q].get(kx);
                    vr[q].get(vx);
                    st8(&sm.kc[t][i], kx);
                    st8(&sm.vv[t][i], vx);
#pragma unroll
                    for (int u = 0; u < 8; u++) ss = fmaf(kx[u], kx[u], ss);
                }
#pragma unroll
                for (int o = 1; o < TPT; o <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                if (in && i == 0) sm.RK[t].y = sqrtf(ss);
            }
        }
    }
    if (own) {
        sm.kap[tid] = okey(kapv);
        sm.RK[tid].x = rtv;
    }
    if (resume && tid < nn && rec_p >= 0) rec_kin = A.nd_kappa[rec_p];
    // thread (pp, c) owns probes pp and pp + 32, elements 4 c + 32 g + j; the
    // 8 chunk lanes of a pair read 128 contiguous bytes
    const int c = lane / kPPW, pp = dwarp * kPPW + (lane & (kPPW - 1));
    auto qrow = [&](int u) -> size_t { return ((size_t)l * A.Hq + g * A.gq + (u % A.gq)) * A.W + u; };
    auto load_q = [&](float2 *qd, int u) {   // the thread's chunk of probe u's query as element pairs
        if (u < A.W) {
            const Tin *qp = static_cast<const Tin *>(A.Q) + qrow(u) * DH + 4 * c;
#pragma unroll
            for (int gi = 0; gi < NG; gi++) {
                const float4 x = ld4(qp + 32 * gi);
                qd[2 * gi] = make_float2(x.x, x.y);
                qd[2 * gi + 1] = make_float2(x.z, x.w);
            }
        } else {
#pragma unroll
            for (int q = 0; q < CH / 2; q++) qd[q] = make_float2(0.f, 0.f);
        }
    };
    // logits: the lane's reduced value belongs to probe pp + 32 (c / 4); the
    // candidate sums: lane p of a warp takes the probes p and p + 32
    const int ulog = pp + kNPP * (c >> 2);
    const float mu_log = ulog < A.W ? A.row_m[qrow(ulog)] : 0.f;
    const float invZ0 = lane < A.W ? 1.0f / A.row_Z[qrow(lane)] : 0.f;
    const float invZ1 = lane + kNPP < A.W ? 1.0f / A.row_Z[qrow(lane + kNPP)] : 0.f;
    // ---- E[t][u] ---------------------------------------------------------------
    if (A.Eg) {
        cp_async_wait<0>();   // the thread's own copies have landed
        for (int idx = tid; idx < n * (2 * kNPP / 4); idx += NT) {
            const float4 e = reinterpret_cast<const float4 *>(Ef)[idx];
            bad |= !(isfinite(e.x) && isfinite(e.y) && isfinite(e.z) && isfinite(e.w));
        }
    } else if constexpr (std::is_same<Tin, __nv_bfloat16>::value) {
        // Tensor cores: logits = Q_probes (64 x DH) . K_slot^T, one 16x8 tile
        // per (probe block, token block); warp w keeps probe block w % 4.
        __syncthreads();   // the raw keys
        constexpr int MT = 4, WSTEP = NWARPS / MT;
        const int gr = lane >> 2, c2 = 2 * (lane & 3);
        const int mt = warp % MT;
        const int u0 = mt * 16 + gr, u1 = u0 + 8;
        const __nv_bfloat16 *Qb = static_cast<const __nv_bfloat16 *>(A.Q);
        const size_t r0 = ((size_t)l * A.Hq + g * A.gq + u0 % A.gq) * A.W + u0;
        const size_t r1 = ((size_t)l * A.Hq + g * A.gq + u1 % A.gq) * A.W + u1;
        const bool ok0 = u0 < A.W, ok1 = u1 < A.W;
        uint32_t qa[DH / 16][4];
#pragma unroll
        for (int ks = 0; ks < DH / 16; ks++) {
            const __nv_bfloat16 *p0 = Qb + r0 * DH + ks * 16 + c2, *p1 = Qb + r1 * DH + ks * 16 + c2;
            qa[ks][0] = ok0 ? *reinterpret_cast<const uint32_t *>(p0) : 0u;
            qa[ks][1] = ok1 ? *reinterpret_cast<const uint32_t *>(p1) : 0u;
            qa[ks][2] = ok0 ? *reinterpret_cast<const uint32_t *>(p0 + 8) : 0u;
            qa[ks][3] = ok1 ? *reinterpret_cast<const uint32_t *>(p1 + 8) : 0u;
        }
        const float m0 = ok0 ? A.row_m[r0] : 0.f, m1 = ok1 ? A.row_m[r1] : 0.f;
        const int ntn = (n + 7) / 8;
        for (int nt = warp / MT; nt < ntn; nt += WSTEP) {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            const float *kr = &sm.kc[tile_row<NMAX>(nt * 8 + gr, n)][c2];
#pragma unroll
            for (int ks = 0; ks < DH / 16; ks++) {
                const float2 x0 = *reinterpret_cast<const float2 *>(kr + ks * 16);
                const float2 x1 = *reinterpret_cast<const float2 *>(kr + ks * 16 + 8);
                mma_bf16(acc, qa[ks], pack_bf16x2(x0.x, x0.y), pack_bf16x2(x1.x, x1.y));
            }
            const int t0 = nt * 8 + c2;
            if (t0 < n) {
                Ef[eidx(t0, u0)] = ok0 ? expf(acc[0] * A.inv_sqrt_d - m0) : 0.f;
                Ef[eidx(t0, u1)] = ok1 ? expf(acc[2] * A.inv_sqrt_d - m1) : 0.f;
            }
            if (t0 + 1 < n) {
                Ef[eidx(t0 + 1, u0)] = ok0 ? expf(acc[1] * A.inv_sqrt_d - m0) : 0.f;
                Ef[eidx(t0 + 1, u1)] = ok1 ? expf(acc[3] * A.inv_sqrt_d - m1) : 0.f;
            }
        }
    } else {
        __syncthreads();   // the raw keys
        float2 qa0[CH / 2], qa1[CH / 2];
        load_q(qa0, pp);
        load_q(qa1, pp + kNPP);
        const float mu0 = pp < A.W ? A.row_m[qrow(pp)] : 0.f;
        const float mu1 = pp + kNPP < A.W ? A.row_m[qrow(pp + kNPP)] : 0.f;
        for (int t = DIRS == 2 ? warp / (kNT / 32) : 0; t < n; t += DIRS) {
            float2 x0 = make_float2(0.f, 0.f), x1 = make_float2(0.f, 0.f);
#pragma unroll
            for (int gi = 0; gi < NG; gi++) {
                const float4 kv = *reinterpret_cast<const float4 *>(&sm.kc[t][4 * c + 32 * gi]);
                const float2 ka = make_float2(kv.x, kv.y), kb = make_float2(kv.z, kv.w);
                x0 = ffma2(qa0[2 * gi], ka, x0); x0 = ffma2(qa0[2 * gi + 1], kb, x0);
                x1 = ffma2(qa1[2 * gi], ka, x1); x1 = ffma2(qa1[2 * gi + 1], kb, x1);
            }
            float y0 = x0.x + x0.y, y1 = x1.x + x1.y;
#pragma unroll
            for (int o = kPPW; o < 32; o <<= 1) {   // over the pair's chunk lanes
                y0 += __shfl_xor_sync(0xffffffffu, y0, o);
                y1 += __shfl_xor_sync(0xffffffffu, y1, o);
            }
            if (c == 0)
                sm.E[t][pp] = make_float2(pp < A.W ? expf(y0 * A.inv_sqrt_d - mu0) : 0.f,
                                          pp + kNPP < A.W ? expf(y1 * A.inv_sqrt_d - mu1) : 0.f);
        }
    }
    if (!A.Eg) {
        __syncthreads();
        for (int e = tid; e < n * 2 * kNPP; e += NT) bad |= !isfinite(Ef[e]);
    }
    // Non-finite probe weights or token values (NaN/Inf in K, Q or the row
    // statistics) make every decision of the unit meaningless: record the
    // unit as a single uncovered leaf with zero gain and flag the error, which
    // the host reports as GKV_ENONFINITE at the allocation's count sync.
    {
        if (__syncthreads_or(bad)) {
            if constexpr (SUB) {   // the node stays a leaf; the unit is reported
                if (tid == 0) {
                    atomicOr(A.status, 8);
                    A.nd_nchild[gv_sub] = 0; A.nd_child0[gv_sub] = -1; A.nd_cost[gv_sub] = 0;
                    A.nd_U[gv_sub] = 0.f; A.nd_kappa[gv_sub] = 0.f;
                }
                return;
            }
            if (tid == 0) {
                atomicOr(A.status, 8);
                A.nd_a[nbase] = sa; A.nd_b[nbase] = sb; A.nd_R[nbase] = 0.f; A.nd_D[nbase] = 0.f;
                A.nd_parent[nbase] = (int32_t)(-2 - uid); A.nd_unit[nbase] = (int32_t)uid;
                A.nd_child0[nbase] = -1; A.nd_nchild[nbase] = 0; A.nd_U[nbase] = 0.f;
                A.nd_kappa[nbase] = 0.f; A.nd_sel[nbase] = 0;
                A.u_nnodes[uid] = 1; A.u_Uadd[uid] = 0.f; A.u_Ddrop[uid] = 0.f; A.u_sel[uid] = 0;
                A.u_pend[uid] = -1.f;
            }
            for (int k = tid; k < 2 * n; k += NT) A.nd_cost[nbase + k] = 0;
            return;
        }
    }
    // Singleton floor (App. A.5 Stage I): the accepted positions of this slot
    // and their scores; a node holding one is extracted at the one of largest
    // score, and the floor's ops carry the largest key (they execute first).
    bool ufl = false;
    if (A.fl_acc) {
        bool any = false;
        for (int t = tid; t < n; t += NT) {
            const size_t q = (size_t)lg * A.Nc + (sa - A.cs) + t;
            const bool ac = A.fl_acc[q] != 0;
            sm.Ff[t] = ac ? A.fl_f[q] : -INFINITY;
            any |= ac;
        }
        ufl = __syncthreads_or(any);
    }
    // ---- k_circ = RoPE^-1(k, t), where the raw keys were needed ----------------
    if (!rotated) {
        constexpr int RB = 4;   // rotation-table loads issued before any is used
        for (int e0 = tid; e0 < n * HALF; e0 += NT * RB) {
            float2 cs[RB];
#pragma unroll
            for (int q = 0; q < RB; q++) {
                const int e = e0 + q * NT;
                if (e < n * HALF) {
                    const int t = e / HALF, i = e - t * HALF;
                    cs[q] = A.rope[(size_t)(sa + t) * HALF + i];
                }
            }
#pragma unroll
            for (int q = 0; q < RB; q++) {
                const int e = e0 + q * NT;
                if (e < n * HALF) {
                    const int t = e / HALF, i = e - t * HALF;
                    const float x = sm.kc[t][i], y = sm.kc[t][i + HALF];
                    rotate_back(x, y, cs[q].x, cs[q].y, sm.kc[t][i], sm.kc[t][i + HALF]);
                }
            }
        }
    }
    // ---- curvature order of the slot's tokens (ties: lower t first), once for all nodes
    // Four threads count a token's predecessors.  A node's candidates then
    // follow from bit masks over these places; counting per node, on the
    // node's own warp, was a serial chain of n^2 / 32 comparisons (skew 64K at
    // 32x, slots of up to 128 tokens: 234.5 -> 223.9 ms; llama128k 90.2 -> 89.2).
    {
        static_assert(NT / 4 >= NMAX && NMAX <= 256, "four threads per token");
        const int t = tid >> 2;
        int before = 0;
        if (t < n) {
            const unsigned long long kt = sm.kap[t];
            for (int q = tid & 3; q < n; q += 4) {
                const unsigned long long kq = sm.kap[q];
                before += (kq > kt) || (kq == kt && q < t);
            }
        }
        before += __shfl_xor_sync(0xffffffffu, before, 1);
        before += __shfl_xor_sync(0xffffffffu, before, 2);
        if (t < n && (tid & 3) == 0) sm.rk[t] = (uint8_t)before;
    }
    // ---- tree state: a fresh root, a subtree's root, or the unit's records so far
    if constexpr (SUB) {
        if (tid == 0) {
            NodeS &nd = sm.nodes[0];
            nd.a = 0; nd.b = (short)n; nd.nchild = -1;
            nd.D = A.nd_D[gv_sub];
            const int32_t pg = A.nd_parent[gv_sub];   // a node of the long unit, already evaluated
            nd.kin = pg < 0 ? FLT_MAX : A.nd_kappa[pg];
            sm.pend = -1.f;
        }
        if (tid < S::MW) sm.lvl[0][tid] = tid == 0 ? 1u : 0u;
        nn = 1;
    } else if (!resume) {
        if (warp == 0) {
            float r = 0.f;
            for (int t = lane; t < n; t += 32) r += sm.RK[t].x;
            r = warp_sum(r);
            if (lane == 0) {
                NodeS &nd = sm.nodes[0];
                nd.a = 0; nd.b = (short)n; nd.nchild = 0;
                nd.D = 0.f; nd.kin = 0.f;
                sm.rootR = r;
                sm.pend = -1.f;
                A.nd_a[nbase] = sa; A.nd_b[nbase] = sb; A.nd_R[nbase] = (float)r;
                A.nd_parent[nbase] = (int32_t)(-2 - uid);
                A.nd_unit[nbase] = (int32_t)uid;
            }
        }
        if (tid < S::MW) sm.lvl[0][tid] = tid == 0 ? 1u : 0u;
        nn = 1;
    } else {
        // the pending nodes whose key bound reaches tau form the first level
        if (tid == 0) sm.pend = -1.f;
        __syncthreads();
        bool q = false;
        if (tid < nn) {
            NodeS &nd = sm.nodes[tid];
            nd.a = (short)(rec_a - sa);
            nd.b = (short)(rec_b - sa);
            nd.nchild = (signed char)rec_nch;
            nd.D = rec_D;
            nd.kin = rec_p < 0 ? (ufl ? FLT_MAX : A.u_Uadd[uid]) : rec_kin;
            if (rec_nch == -1) {   // nd_U holds the key bound of a pending node
                q = rec_U >= A.tau;
                if (!q) atomicMax(reinterpret_cast<int *>(&sm.pend), __float_as_int(rec_U));
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, q);
        if (lane == 0 && warp < S::MW) sm.lvl[0][warp] = m;
    }
    // a fresh root's attention mass, mean over the probes, where it decides how the
    // root is evaluated (thread tid adds the tokens' weights of one probe)
    const bool weigh = fresh && !A.root_only && A.prune && A.lam_kappa > 0.f && A.lam_kappa < kDirectMax;
    if (weigh) {
        const int e0 = tid & (2 * kNPP - 1), u = (e0 >> 1) + kNPP * (e0 & 1);
        float p = 0.f;
        for (int e = tid; e < n * 2 * kNPP; e += NT) p += Ef[e];
        p = warp_sum(u < A.W ? p / A.row_Z[qrow(u)] : 0.f);
        if (lane == 0) sm.candP[warp] = p;
    }
    __syncthreads();
    float mass = 0.f;
    if (weigh) {
        for (int w = 0; w < NWARPS; w++) mass += sm.candP[w];
        mass /= A.W;
    }

    unsigned int w_scan = 0, w_eval = 0, w_len = 0;   // work counters (lane 0 of each warp)

    // Prototype (ktil, vtil, m_eff) of one or two candidate rows: row r0, and r1
    // (-1: none), either two prefixes of a node (ascending ends; one running
    // sum gives both) or two suffixes (descending starts; one set of loads
    // feeds both sums).  Every sum runs over its interval's tokens in
    // ascending order.  The keys' and the values' sums are separate tasks, so
    // that a lone node keeps several warps busy.
    constexpr int PPL = HALF / 32;   // rotation pairs per lane: (i, i + d/2), i = PPL lane + j
    const int pi0 = lane * PPL;
    auto proto_keys = [&](int r0, int r1, auto SUF) {
        constexpr bool suffix = decltype(SUF)::value;
        // the 64-channel bf16 instances' prefixes fuse the other product (their bits since the first build)
        constexpr bool SF = DH == 64 && std::is_same<Tin, __nv_bfloat16>::value && !SUB && !suffix;
        using PS = KeySum<PPL, HALF>;
        const int a0 = sm.cand[r0].a, b0 = sm.cand[r0].b;
        const int a1 = r1 >= 0 ? sm.cand[r1].a : 0, b1 = r1 >= 0 ? sm.cand[r1].b : 0;
        float2 rot0[PPL], rot1[PPL];   // loaded first, so that their latency overlaps the sums
        const int p0 = round_half_even_mid(sa + a0, sa + b0), p1 = round_half_even_mid(sa + a1, sa + b1);
#pragma unroll
        for (int j = 0; j < PPL; j++) {
            rot0[j] = A.rope[(size_t)p0 * HALF + pi0 + j];
            rot1[j] = r1 >= 0 ? A.rope[(size_t)p1 * HALF + pi0 + j] : make_float2(0.f, 0.f);
        }
        auto put = [&](int row, int nJ, const float2 *rot, const PS &acc) {
            const float ninv = 1.0f / (float)nJ;
            float mu2 = 0.f;
#pragma unroll
            for (int j = 0; j < PPL; j++) {
                const float a0 = acc.lo(j) * ninv, a1 = acc.hi(j) * ninv;
                mu2 = fmaf(a0, a0, fmaf(a1, a1, mu2));
                const float2 cs = rot[j];
                rotate_to<SF>(a0, a1, cs.x, cs.y, sm.ktil(row)[pi0 + j], sm.ktil(row)[pi0 + j + HALF]);
            }
            mu2 = warp_sum(mu2);
            if (lane == 0) {
                const float coh = sqrtf(mu2) / (acc.ks * ninv + A.eps);
                const float me = (float)nJ * coh * coh;
                sm.cand[row].meff = me < 1.0f ? 1.0f : (me > (float)nJ ? (float)nJ : me);
            }
        };
        PS s0;
        s0.clear();
        if (!suffix) {
#pragma unroll 4
            for (int t = a0; t < b0; t++) s0.add(&sm.kc[t][pi0], sm.RK[t].y);
            put(r0, b0 - a0, rot0, s0);
            if (r1 < 0) return;
#pragma unroll 4
            for (int t = b0; t < b1; t++) s0.add(&sm.kc[t][pi0], sm.RK[t].y);
            put(r1, b1 - a1, rot1, s0);
        } else {
            PS s1;
            s1.clear();
            if (r1 >= 0) {   // the longer one's own tokens
#pragma unroll 4
                for (int t = a1; t < a0; t++) s1.add(&sm.kc[t][pi0], sm.RK[t].y);
#pragma unroll 4
                for (int t = a0; t < b0; t++) {
                    s0.add(&sm.kc[t][pi0], sm.RK[t].y);
                    s1.add(&sm.kc[t][pi0], sm.RK[t].y);
                }
                put(r1, b1 - a1, rot1, s1);
            } else {
#pragma unroll 4
                for (int t = a0; t < b0; t++) s0.add(&sm.kc[t][pi0], sm.RK[t].y);
            }
            put(r0, b0 - a0, rot0, s0);
        }
    };
    auto proto_values = [&](int r0, int r1, auto SUF) {
        constexpr bool suffix = decltype(SUF)::value;
        using PS = ValueSum<PPL, HALF>;
        const int a0 = sm.cand[r0].a, b0 = sm.cand[r0].b;
        const int a1 = r1 >= 0 ? sm.cand[r1].a : 0, b1 = r1 >= 0 ? sm.cand[r1].b : 0;
        auto put = [&](int row, int nJ, const PS &acc) {
            const float ninv = 1.0f / (float)nJ;
            const float beta = (float)A.base_frac * (acc.rs * ninv);
            const float winv = 1.0f / ((acc.rs + (float)nJ * beta) + A.eps);
#pragma unroll
            for (int j = 0; j < PPL; j++) {
                sm.vtil(row)[pi0 + j] = fmaf(beta, acc.slo(j), acc.rlo(j)) * winv;
                sm.vtil(row)[pi0 + j + HALF] = fmaf(beta, acc.shi(j), acc.rhi(j)) * winv;
            }
        };
        PS s0;
        s0.clear();
        if (!suffix) {
#pragma unroll 4
            for (int t = a0; t < b0; t++) s0.add(&sm.vv[t][pi0], sm.RK[t].x);
            put(r0, b0 - a0, s0);
            if (r1 < 0) return;
#pragma unroll 4
            for (int t = b0; t < b1; t++) s0.add(&sm.vv[t][pi0], sm.RK[t].x);
            put(r1, b1 - a1, s0);
        } else {
            PS s1;
            s1.clear();
            if (r1 >= 0) {
#pragma unroll 4
                for (int t = a1; t < a0; t++) s1.add(&sm.vv[t][pi0], sm.RK[t].x);
#pragma unroll 2
                for (int t = a0; t < b0; t++) {
                    s0.add(&sm.vv[t][pi0], sm.RK[t].x);
                    s1.add(&sm.vv[t][pi0], sm.RK[t].x);
                }
                put(r1, b1 - a1, s1);
            } else {
#pragma unroll 4
                for (int t = a0; t < b0; t++) s0.add(&sm.vv[t][pi0], sm.RK[t].x);
            }
            put(r0, b0 - a0, s0);
        }
    };
    // The prototypes of the rows [rb, re) of one direction (one node's), two
    // at a time; `task` counts the tasks handed out, round robin over the warps.
    auto prototypes = [&](int rb, int re, auto SUF, int &task) {
        for (int r = rb; r < re; r += 2) {
            const int r1 = r + 1 < re ? r + 1 : -1;
            if (task++ % NWARPS == warp) proto_keys(r, r1, SUF);
            if (task++ % NWARPS == warp) proto_values(r, r1, SUF);
        }
    };
    const float inv_sqrt_d = A.inv_sqrt_d, lamZ = A.lamZ, lamM = A.lamM, epsf = A.eps;
    // zt = m_eff exp(q_u . ktil / sqrt d - m_u) of the rows [0, nr), four at a
    // time: 8 dot products per thread chunk, one reduce-scatter, and one
    // exponential per (row, probe).  Starts with the barrier that the
    // prototypes end on, after the queries' loads.
    auto logits = [&](int nr) {
        float2 qa0[CH / 2], qa1[CH / 2];
        load_q(qa0, pp);
        load_q(qa1, pp + kNPP);
        __syncthreads();
        for (int i = DIRS == 2 ? 4 * (warp / (kNT / 32)) : 0; i < nr; i += 4 * DIRS) {
            float v[8];   // [row i + (index & 3)][probe pp + 32 (index >> 2)]
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int row = min(i + j, nr - 1);
                float2 xa = make_float2(0.f, 0.f), xb = make_float2(0.f, 0.f);
#pragma unroll
                for (int gi = 0; gi < NG; gi++) {
                    const float4 x = *reinterpret_cast<const float4 *>(&sm.ktil(row)[4 * c + 32 * gi]);
                    const float2 ka = make_float2(x.x, x.y), kb = make_float2(x.z, x.w);
                    xa = ffma2(qa0[2 * gi], ka, xa);
                    xa = ffma2(qa0[2 * gi + 1], kb, xa);
                    xb = ffma2(qa1[2 * gi], ka, xb);
                    xb = ffma2(qa1[2 * gi + 1], kb, xb);
                }
                v[j] = xa.x + xa.y;
                v[4 + j] = xb.x + xb.y;
            }
            const float x = reduce_scatter8(v, lane);
            const int row = i + (c & 3);
            if (row < nr)
                reinterpret_cast<float *>(&sm.zt(row)[pp])[c >> 2] =
                    sm.cand[row].meff * expf(x * inv_sqrt_d - mu_log);
        }
    };
    // Probe scan of one node in one direction (SUF: suffixes, descending):
    // running sums Z_u, M_u over the tokens from position t0; at the far end of
    // each of the rows [k, ke) the thread's parts of ||M - zt vtil||^2 and
    // ||M||^2 are reduced, and their ratio and Z go into the row's (no longer
    // needed) key prototype.
    auto scan = [&](int t0, int k, int ke, auto SUF) {
        constexpr bool suffix = decltype(SUF)::value;
        if (k >= ke) return;
        int t = t0;   // next token to add
        float2 M0[CH / 2], M1[CH / 2];
        float2 Z = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < CH / 2; q++) M0[q] = M1[q] = make_float2(0.f, 0.f);
        auto add = [&](int t) {
            const float2 e = sm.E[t][pp];
            const float2 e0 = make_float2(e.x, e.x), e1 = make_float2(e.y, e.y);
            Z = fadd2(Z, e);
#pragma unroll
            for (int gi = 0; gi < NG; gi++) {
                const float4 x = *reinterpret_cast<const float4 *>(&sm.vv[t][4 * c + 32 * gi]);
                const float2 va = make_float2(x.x, x.y), vb = make_float2(x.z, x.w);
                M0[2 * gi] = ffma2(e0, va, M0[2 * gi]);
                M0[2 * gi + 1] = ffma2(e0, vb, M0[2 * gi + 1]);
                M1[2 * gi] = ffma2(e1, va, M1[2 * gi]);
                M1[2 * gi + 1] = ffma2(e1, vb, M1[2 * gi + 1]);
            }
        };
        for (; k < ke; k++) {
            if (suffix) {
                const int stop = sm.cand[k].a;   // rows in descending start
#pragma unroll 2
                for (; t >= stop; t--) add(t);
            } else {
                const int stop = sm.cand[k].b;   // rows in ascending end
#pragma unroll 2
                for (; t < stop; t++) add(t);
            }
            const float2 z = sm.zt(k)[pp];
            const float2 nz0 = make_float2(-z.x, -z.x), nz1 = make_float2(-z.y, -z.y);
            float2 r0 = make_float2(0.f, 0.f), r1 = r0, m0 = r0, m1 = r0;
#pragma unroll
            for (int gi = 0; gi < NG; gi++) {
                const float4 x = *reinterpret_cast<const float4 *>(&sm.vtil(k)[4 * c + 32 * gi]);
                const float2 va = make_float2(x.x, x.y), vb = make_float2(x.z, x.w);
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int q = 2 * gi + h;
                    const float2 vt = h ? vb : va;
                    const float2 d0 = ffma2(nz0, vt, M0[q]), d1 = ffma2(nz1, vt, M1[q]);   // M - zt vtil
                    r0 = ffma2(d0, d0, r0);
                    r1 = ffma2(d1, d1, r1);
                    m0 = ffma2(M0[q], M0[q], m0);
                    m1 = ffma2(M1[q], M1[q], m1);
                }
            }
            // lane c: probe pp + 32 (c & 1), ||M||^2 if c & 2 else the residual;
            // the residual's lane divides, its partner keeps Z.  Fast division:
            // at most 2 ulp, far below the distortion tolerance.
            const float x = reduce_scatter4(r0.x + r0.y, r1.x + r1.y, m0.x + m0.y, m1.x + m1.y, lane);
            const float y = __shfl_xor_sync(0xffffffffu, x, 2 * kPPW);
            if (c < 4) sm.ktil(k)[4 * pp + c] = (c & 2) ? ((c & 1) ? Z.y : Z.x) : __fdividef(x, y + epsf);
        }
    };
    // D_u (Eq. app_probe_distortion) of the rows [0, nr), weighted by the
    // probe's attention mass, and their means over the W probes: a warp per
    // row, lane p the probes p and p + 32.  The sums run over groups of four
    // lanes, then over the groups in order.  Probes past W have E = 0 and
    // invZ = 0, so they add nothing.
    auto finish = [&](int nr, int out) {
        const float invW = 1.0f / A.W;
        for (int k = warp; k < nr; k += NWARPS) {
            if (sm.cand[k].b <= sm.cand[k].a) continue;
            const float4 q = *reinterpret_cast<const float4 *>(&sm.ktil(k)[4 * lane]);   // ratios, Z
            const float2 z = sm.zt(k)[lane];
            const float Z0 = q.z, Z1 = q.w;
            const float dz0 = Z0 - z.x, dz1 = Z1 - z.y;
            const float D0 = fmaf(lamZ, __fdividef(dz0 * dz0, fmaf(Z0, Z0, epsf)), lamM * q.x);
            const float D1 = fmaf(lamZ, __fdividef(dz1 * dz1, fmaf(Z1, Z1, epsf)), lamM * q.y);
            const float p0 = Z0 * invZ0, p1 = Z1 * invZ1;
            float pd = fmaf(p0, D0, p1 * D1), pw = p0 + p1;
#pragma unroll
            for (int o = 1; o < kPPW; o <<= 1) {
                pd += __shfl_xor_sync(0xffffffffu, pd, o);
                pw += __shfl_xor_sync(0xffffffffu, pw, o);
            }
            const float x = (lane & 1) ? pw : pd;   // even lanes sum D, odd lanes the mass
            float d = 0.f;
#pragma unroll
            for (int w = 0; w < 32 / kPPW; w++) d += __shfl_sync(0xffffffffu, x, kPPW * w + (lane & 1));
            if (lane < 2) (lane ? sm.candP : sm.candD)[out + k] = d * invW;
        }
    };

    // A fresh root's D, Ddrop and Add gain (Eq. app_operation_gains), from its own row.
    auto root_done = [&](NodeS &nd, int row) {
        const float Pd = sm.candP[row];
        const float D = nd.b - nd.a >= 2 ? sm.candD[row] : 0.f;
        nd.D = D;
        float gain = om * sm.rootR * (Pd - D);
        if (gain < 0.f) gain = 0.f;
        nd.kin = ufl ? FLT_MAX : gain;   // a floor slot's Add is a floor op
        A.u_Uadd[uid] = gain;
        A.u_Ddrop[uid] = Pd;
        A.nd_D[gidx(0)] = D;
    };
    // The cuts of an open node, one per lane, and its rows: prefixes of the cuts
    // in B.more and of the extraction by ascending end (then a direct root
    // itself), suffixes of the cuts in B.keep by descending start.
    struct Open {
        int a, b, ps, xi, prow, srow, el_row, er_row;   // rows relative to the node's first of a direction
        float rew;
        bool pv, sv, el, er, elr, err;   // el, er: the extraction's sides; elr, err: in rows of their own
    };
    auto open_rows = [&](const BatchNode &B) {
        const unsigned FULL = 0xffffffffu, lt = (1u << lane) - 1u, gt = ~((2u << lane) - 1u);
        const NodeS &nd = sm.nodes[B.node];
        Open o;
        o.a = nd.a;
        o.b = nd.b;
        o.ps = B.pstar;
        o.xi = lane < B.ncut ? B.cut[lane] : 0;
        o.rew = lane < B.ncut ? B.kh[lane] : 0.f;
        o.pv = ((B.more >> lane) & 1u) && o.xi - o.a >= 2;
        o.sv = ((B.keep >> lane) & 1u) && o.b - o.xi >= 2;
        o.el = B.ext && o.ps - o.a >= 2;
        o.er = B.ext && o.b - (o.ps + 1) >= 2;
        // a side equal to a cut's shares its row
        o.elr = o.el && !__any_sync(FULL, o.pv && o.xi == o.ps);
        o.err = o.er && !__any_sync(FULL, o.sv && o.xi == o.ps + 1);
        o.prow = __popc(__ballot_sync(FULL, o.pv) & lt) + (o.elr && o.ps < o.xi ? 1 : 0);
        o.srow = __popc(__ballot_sync(FULL, o.sv) & gt) + (o.err && o.ps + 1 > o.xi ? 1 : 0);
        o.el_row = __popc(__ballot_sync(FULL, o.pv && o.xi < o.ps));
        o.er_row = __popc(__ballot_sync(FULL, o.sv && o.xi > o.ps + 1));
        return o;
    };
    auto best_first = [&](const BatchNode &B) {   // G_bin of the cut evaluated ahead
        return B.direct ? -INFINITY : fmaf(A.lam_kappa, B.kh[B.k1], (sm.nodes[B.node].D - B.cD[0]) - B.cD[1]);
    };
    // The decision over all cuts that no bound ruled out, ties to the smallest xi.
    auto decide_open = [&](BatchNode &B, int sufD) {
        const unsigned FULL = 0xffffffffu;
        const Open o = open_rows(B);
        const float DI = sm.nodes[B.node].D, best1 = best_first(B);
        const int ncut = B.ncut;
        float dl = o.pv ? sm.candD[B.pre_b + o.prow] : 0.f, dr = o.sv ? sm.candD[sufD + B.suf_b + o.srow] : 0.f;
        // a cut ruled out keeps a bound below best1
        float val = -INFINITY;
        if (!B.direct && lane == B.k1) { dl = B.cD[0]; dr = B.cD[1]; val = best1; }
        else if ((B.keep >> lane) & 1u) val = fmaf(A.lam_kappa, o.rew, (DI - dl) - dr);
        const unsigned key = lane < ncut ? fkey_ordered(val) : 0u;
        const unsigned kmx = __reduce_max_sync(FULL, key);   // every lane takes part
        const unsigned top = __ballot_sync(FULL, lane < ncut && key == kmx);
        int bq = __ffs(top) - 1;
        const float best = __shfl_sync(FULL, val, bq);
        if (!(best > -INFINITY)) bq = 0;   // only reachable with non-finite gains
        const float bL = __shfl_sync(FULL, dl, bq), bR = __shfl_sync(FULL, dr, bq);
        if (lane) return;
        const float eDL = o.el ? sm.candD[B.pre_b + o.el_row] : 0.f, eDR = o.er ? sm.candD[sufD + B.suf_b + o.er_row] : 0.f;
        bool take = false;
        if (B.ext) {   // rho_ext = G_ext / (|children| - 1)
            const int ne = 1 + (o.ps > o.a) + (o.ps + 1 < o.b);
            float gext = DI;
            if (o.ps > o.a) gext -= eDL;
            if (o.ps + 1 < o.b) gext -= eDR;
            take = (ne == 3 ? 0.5f * gext : gext) > best;
        }
        if (take) {
            set_extraction(B, o.a, o.b, eDL, eDR);
        } else {
            B.nchild = 2;
            B.ca[0] = (short)o.a; B.cb[0] = B.cut[bq]; B.cD[0] = bL;
            B.ca[1] = B.cut[bq]; B.cb[1] = (short)o.b; B.cD[1] = bR;
        }
    };
    // D_L of a node's prefixes known: the cuts that need no suffix drop out.
    auto narrow_open = [&](BatchNode &B) {
        const Open o = open_rows(B);
        const float dl = o.pv ? sm.candD[B.pre_b + o.prow] : 0.f;
        bool need = (B.more >> lane) & 1u;
        if (need && A.prune) need = !(fmaf(A.lam_kappa, o.rew, sm.nodes[B.node].D - dl) < best_first(B));
        const unsigned keep = __ballot_sync(0xffffffffu, need);
        const bool err = o.er && !__any_sync(0xffffffffu, need && o.xi == o.ps + 1);
        const int ns = __popc(__ballot_sync(0xffffffffu, need && o.b - o.xi >= 2)) + err;
        if (lane == 0) {
            B.keep = keep;
            B.ns = (int8_t)ns;
        }
    };
    // The rows of an open node from row r on: np prefixes, then ns suffixes (0: none now).
    auto lay_out = [&](BatchNode &B, int r, int np, int ns, bool pre) {
        const Open o = open_rows(B);
        if (np && o.pv) sm.cand[r + o.prow] = {(short)o.a, (short)o.xi, 0.f};
        if (ns && o.sv) sm.cand[r + np + o.srow] = {(short)o.xi, (short)o.b, 0.f};
        int len = (np && o.pv ? o.xi - o.a : 0) + (ns && o.sv ? o.b - o.xi : 0);
        int pe = np && o.pv ? o.xi : o.a, ss = ns && o.sv ? o.xi : o.b;
        len = __reduce_add_sync(0xffffffffu, len);
        pe = __reduce_max_sync(0xffffffffu, pe);
        ss = __reduce_min_sync(0xffffffffu, ss);
        if (lane == 0) {
            if (np && o.elr) {
                sm.cand[r + o.el_row] = {(short)o.a, (short)o.ps, 0.f};
                pe = max(pe, o.ps);
                len += o.ps - o.a;
            }
            if (ns && o.err) {
                sm.cand[r + np + o.er_row] = {(short)(o.ps + 1), (short)o.b, 0.f};
                ss = min(ss, o.ps + 1);
                len += o.b - o.ps - 1;
            }
            if (np && B.direct && B.node == 0 && fresh) {
                sm.cand[r + np - 1] = {(short)o.a, (short)o.b, 0.f};
                pe = o.b;
                len += o.b - o.a;
            }
            if (pre) { B.pre_b = (int8_t)r; B.pre_e = (int8_t)(r + np); }   // kept while the suffixes follow
            B.suf_b = (int8_t)(r + np);
            B.suf_e = (int8_t)(r + np + ns);
            w_scan += (pe - o.a) + (o.b - ss);
            w_eval += np + ns;
            w_len += len;
        }
    };

    int cur = 0;
    for (int levels_left = A.max_levels;; cur ^= 1) {
        unsigned any = 0;
        for (int w = 0; w < S::MW; w++) any |= sm.lvl[cur][w];
        if (!any) break;
        levels_left--;   // the last level's children stay pending (D2)
        if (tid < S::MW) sm.lvl[cur ^ 1][tid] = 0;
        int lw = 0;
        unsigned lbits = sm.lvl[cur][0];
        for (;;) {
            // ---- batch: the level's next nodes in creation order.  Every warp
            // walks them; phase A (cut candidates) runs on a node's own warp.
            int nb = 0, nops = 0, nrow = 0;
            while (nb < S::NB) {
                while (!lbits && lw < S::MW - 1) lbits = sm.lvl[cur][++lw];
                if (!lbits) break;
                const int v = lw * 32 + __ffs(lbits) - 1;
                const int a = sm.nodes[v].a, b = sm.nodes[v].b, nv = b - a;
                const bool root = v == 0 && fresh;
                const bool ronly = root && A.root_only;   // only the node's own distortion
                // no cut is evaluated ahead where the bound could hardly rule another out
                // (floor slots: an extraction may be forced)
                const bool direct = nv >= 3 && !ronly && !ufl &&
                                    !(A.prune && A.lam_kappa > (root ? kDirectRoot * mass : kDirect * sm.nodes[v].D));
                const int rows = direct ? 0 : (nv >= 3 && !ronly ? 2 : 0) + (root ? 1 : 0);
                if (nrow + rows > kNCR) break;
                lbits &= lbits - 1;
                const int row0 = nrow;
                nrow += rows;
                const int op = nv >= 2 && !ronly ? nops++ : -1;
                const int bi = nb++;
                if (bi % NWARPS != warp) continue;
                BatchNode &B = sm.bn[bi];
                // top-K by curvature over positions [a, b-2] (ties: lower t): the
                // places of the node's positions as a bit mask; a position's rank is
                // the number of set places before its own
                constexpr int NW = (NMAX + 31) / 32;
                unsigned sel[NW], places[NW];
                int place[NW];
#pragma unroll
                for (int w = 0; w < NW; w++) {
                    const int t = a + w * 32 + lane;
                    place[w] = !ronly && t <= b - 2 ? (int)sm.rk[t] : -1;
                }
#pragma unroll
                for (int v = 0; v < NW; v++) {
                    unsigned m = 0;
#pragma unroll
                    for (int w = 0; w < NW; w++)
                        if (place[w] >> 5 == v) m |= 1u << (place[w] & 31);
                    places[v] = __reduce_or_sync(0xffffffffu, m);
                }
#pragma unroll
                for (int w = 0; w < NW; w++) {
                    bool s = false;
                    if (place[w] >= 0) {
                        const int t = a + w * 32 + lane;
                        int rank = 0;
#pragma unroll
                        for (int v = 0; v < NW; v++) {
                            const int hi = place[w] - 32 * v;   // places of word v before this one
                            rank += __popc(places[v] & (hi >= 32 ? ~0u : hi <= 0 ? 0u : (1u << hi) - 1u));
                        }
                        if (rank == 0) B.khi = sm.kap[t];
                        if (rank == nv - 2) B.klo = sm.kap[t];
                        s = rank < A.k_cand || t == a + nv / 2 - 1;   // + midpoint
                    }
                    sel[w] = __ballot_sync(0xffffffffu, s);
                }
                // salient token p* = argmax R_tok over [a, b) (ties: lower t)
                float rb = -INFINITY;
                int pb = 0x7fffffff;
                for (int t = a + lane; t < b; t += 32) {
                    const float r = sm.RK[t].x;
                    if (r > rb) { rb = r; pb = t; }
                }
                {
                    const unsigned key = fkey_ordered(rb), kmx = __reduce_max_sync(0xffffffffu, key);
                    pb = __reduce_min_sync(0xffffffffu, key == kmx ? pb : 0x7fffffff);
                }
                if (pb < a || pb >= b) pb = a;   // only reachable with non-finite values
                // a node holding an accepted floor position is extracted at the one
                // of largest floor score (ties: lower t)
                int forced = 0;
                if (ufl) {
                    float fb = -INFINITY;
                    int fpos = 0x7fffffff;
                    for (int t = a + lane; t < b; t += 32) {
                        const float fv = sm.Ff[t];
                        if (fv > fb) { fb = fv; fpos = t; }
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const float f2 = __shfl_xor_sync(0xffffffffu, fb, o);
                        const int p2 = __shfl_xor_sync(0xffffffffu, fpos, o);
                        if (f2 > fb || (f2 == fb && p2 < fpos)) { fb = f2; fpos = p2; }
                    }
                    if (fb > -INFINITY) { pb = fpos; forced = 1; }
                }
                // cuts xi in ascending order, their normalised curvature, and the
                // one of largest reward
                const bool cands = nv >= 3 && !ronly;
                const int maxc = cands ? min(A.k_cand + 1, nv - 1) : 0;
                int ncut = 0;
#pragma unroll
                for (int w = 0; w < (NMAX + 31) / 32; w++) {
                    const unsigned m = sel[w];
                    const int q = ncut + __popc(m & ((1u << lane) - 1u));
                    if (((m >> lane) & 1u) && q < maxc) B.cut[q] = (int8_t)(a + w * 32 + lane + 1);
                    ncut += __popc(m);
                }
                ncut = min(ncut, maxc);
                __syncwarp();
                float rew = 0.f;
                if (lane < ncut) {
                    // the difference is taken in fp64 (the curvatures may be close),
                    // the rest in fp32
                    const double kmn = okey_inv(B.klo), kmx = okey_inv(B.khi);
                    const float krange = kmx > kmn ? 1.0f / (float)(kmx - kmn) : 0.f;
                    const float kh = (float)(okey_inv(sm.kap[B.cut[lane] - 1]) - kmn) * krange;
                    B.kh[lane] = kh;
                    rew = A.lam_kappa * kh;
                }
                const unsigned rkey = lane < ncut ? fkey_ordered(rew) : 0u;
                const int k1 = __ffs(__ballot_sync(0xffffffffu, rkey == __reduce_max_sync(0xffffffffu, rkey))) - 1;
                if (lane == 0) {
                    // the intervals evaluated first: both sides of the cut of largest
                    // reward, or of a forced extraction; a fresh root's own
                    const bool ahead = cands && !direct;
                    const int lo = !ahead ? a : (forced ? pb : B.cut[k1]), hi = !ahead ? b : (forced ? pb + 1 : B.cut[k1]);
                    const bool pv = lo - a >= 2, sv = b - hi >= 2;
                    int k = row0;
                    B.pre_b = (int8_t)k;
                    B.rl = pv ? (int8_t)k : (int8_t)-1;
                    if (pv) sm.cand[k++] = {(short)a, (short)lo, 0.f};
                    const bool own = root && !direct;
                    B.whole = own ? (int8_t)k : (int8_t)-1;
                    if (own) sm.cand[k++] = {(short)a, (short)b, 0.f};
                    B.pre_e = B.suf_b = (int8_t)k;
                    B.rr = sv ? (int8_t)k : (int8_t)-1;
                    if (sv) sm.cand[k++] = {(short)hi, (short)b, 0.f};
                    B.suf_e = (int8_t)k;
                    for (; k < row0 + rows; k++) sm.cand[k].a = sm.cand[k].b = 0;   // reserved, not used
                    B.node = (short)v;
                    B.op = (short)op;
                    B.pstar = (short)pb;
                    B.forced = (int8_t)forced;
                    B.direct = (int8_t)direct;
                    B.ncut = (int8_t)ncut;
                    B.k1 = (int8_t)k1;
                    // work counters: tokens swept, candidates evaluated, their lengths
                    w_scan += (own ? nv : (pv ? lo - a : 0)) + (sv ? b - hi : 0);
                    w_eval += B.suf_e - B.pre_b;
                    w_len += (pv ? lo - a : 0) + (sv ? b - hi : 0) + (own ? nv : 0);
                }
            }
            // the ops' places in the global list, fetched while the batch is evaluated
            if (nops > 0 && tid == NT - 1) sm.op_base = atomicAdd(A.n_ops, (unsigned)nops);
            if (nb == 0) break;
            // Turns: first the rows laid out above, then those of the batch's open
            // nodes (the candidates that the first ones could not rule out), as many
            // nodes at a time as fit the rows: both sides of the cuts in
            // B.more and of the extraction (B.ext).  Their prefixes go first, and the
            // D of those tighten the cuts' bounds before the suffixes follow; both
            // go together when all of them fit.  A node's own warp lays its rows out
            // and decides.  (One open node at a time, with the barriers of a turn
            // each, was slower than evaluating every candidate at once where few
            // cuts are ruled out.)  One loop for all turns keeps one copy of their code.
            unsigned grp = (1u << nb) - 1u, left = 0u;   // the turn's nodes; open ones still to come
            int nr = nrow, dout = 0, lnp = 0, lns = 0;   // lane i: the open node i's candidates
            bool first = true, pre = true, suf = true, dir = false;
            for (;;) {
                __syncthreads();
                // ---- phases B/C: prototypes, logits, scans in both directions, sums --
                if (nr > 0) {
                    int task = 0;
                    for (unsigned m = grp; m; m &= m - 1) {
                        const BatchNode &B = sm.bn[__ffs(m) - 1];
                        if (pre) prototypes(B.pre_b, B.pre_e, std::false_type(), task);
                        if (suf) prototypes(B.suf_b, B.suf_e, std::true_type(), task);
                    }
                    logits(nr);   // after a barrier
                    __syncthreads();
                    for (unsigned m = grp; m; m &= m - 1) {
                        const BatchNode &B = sm.bn[__ffs(m) - 1];
                        const NodeS &nd = sm.nodes[B.node];
                        if (pre && (DIRS == 1 || warp < kNT / 32)) scan(nd.a, B.pre_b, B.pre_e, std::false_type());
                        if (suf && (DIRS == 1 || warp >= kNT / 32)) scan(nd.b - 1, B.suf_b, B.suf_e, std::true_type());
                    }
                    __syncthreads();
                    finish(nr, pre ? 0 : dout);
                    __syncthreads();
                }
                if (first) {
                    // ---- phase D1: decisions (warp per node) ---------------------------------
                    // G_bin of a cut is ((D - D_L) - D_R) + lambda_kappa kh, and D_L, D_R >= 0:
                    // D + lambda_kappa kh bounds it from above, in the rounded arithmetic too
                    // (every operation is monotone; G_bin and its bounds all fuse the
                    // product).  A cut whose bound is below G_bin of the cut already evaluated
                    // cannot be the best one, and its intervals are never evaluated; neither are
                    // the extraction's sides when that G_bin reaches D, which bounds rho_ext.
                    // D of a node is at most its attention mass, so on long contexts the
                    // curvature's reward decides nearly every cut.
                    bool open = false;   // the warp's nodes need more candidates
                    for (int bi = warp; bi < nb; bi += NWARPS) {
                        BatchNode &B = sm.bn[bi];
                        NodeS &nd = sm.nodes[B.node];
                        const int a = nd.a, b = nd.b, nv = b - a;
                        if (B.whole >= 0 && lane == 0) root_done(nd, B.whole);
                        __syncwarp();
                        if (A.root_only && B.whole >= 0 && nv >= 2) {   // its split is decided later
                            if (lane == 0) B.nchild = -1;
                            continue;
                        }
                        if (nv < 3) {
                            if (lane == 0) {
                                B.nchild = 0;
                                if (nv == 2) {
                                    B.nchild = 2;
                                    B.ca[0] = (short)a; B.cb[0] = (short)(a + 1); B.cD[0] = 0.f;
                                    B.ca[1] = (short)(a + 1); B.cb[1] = (short)b; B.cD[1] = 0.f;
                                }
                            }
                            continue;
                        }
                        const float DI = nd.D;
                        const float DL = B.rl >= 0 ? sm.candD[B.rl] : 0.f, DR = B.rr >= 0 ? sm.candD[B.rr] : 0.f;
                        if (B.forced) {
                            if (lane == 0) set_extraction(B, a, b, DL, DR);
                            continue;
                        }
                        bool need = lane < B.ncut, ext = true;
                        if (!B.direct) {
                            const int k1 = B.k1;
                            const float best = fmaf(A.lam_kappa, B.kh[k1], (DI - DL) - DR);
                            need = need && lane != k1;
                            if (need && A.prune) need = !(fmaf(A.lam_kappa, B.kh[lane], DI) < best);
                            ext = !(A.prune && best >= DI);
                            if (lane == 0) {
                                B.ca[0] = (short)a; B.cb[0] = B.cut[k1]; B.cD[0] = DL;
                                B.ca[1] = B.cut[k1]; B.cb[1] = (short)b; B.cD[1] = DR;
                            }
                        }
                        const unsigned more = __ballot_sync(0xffffffffu, need);
                        const bool undecided = more || ext;
                        if (lane == 0) B.nchild = undecided ? -2 : 2;
                        if (!undecided) continue;
                        const int xi = need ? B.cut[lane] : 0;
                        const int ps = B.pstar;
                        const bool elr = ext && ps - a >= 2 && !__any_sync(0xffffffffu, need && xi == ps);
                        const bool err = ext && b - ps - 1 >= 2 && !__any_sync(0xffffffffu, need && xi == ps + 1);
                        const int np = __popc(__ballot_sync(0xffffffffu, need && xi - a >= 2)) + elr +
                                       (B.direct && B.node == 0 && fresh);
                        const int ns = __popc(__ballot_sync(0xffffffffu, need && b - xi >= 2)) + err;
                        if (lane == 0) {
                            B.more = B.keep = more;
                            B.ext = ext;
                            B.np = (int8_t)np;
                            B.ns = (int8_t)ns;
                        }
                        open = true;
                    }
                    if (!__syncthreads_or(open)) break;
                    first = false;
                    const bool op = lane < nb && sm.bn[lane].nchild == -2;
                    left = __ballot_sync(0xffffffffu, op);
                    if (op) { lnp = sm.bn[lane].np; lns = sm.bn[lane].ns; }
                } else {
                    if (pre && fresh && (grp & 1u) && warp == 0 && sm.bn[0].direct && sm.bn[0].node == 0) {
                        if (lane == 0) root_done(sm.nodes[0], sm.bn[0].pre_e - 1);
                        __syncwarp();
                    }
                    if (!suf) {   // the suffixes of the same nodes
                        if (!dir) {   // (direct nodes have no cut yet that could rule one out)
                            for (unsigned m = grp; m; m &= m - 1) {
                                const int bi = __ffs(m) - 1;
                                if (bi % NWARPS == warp) narrow_open(sm.bn[bi]);
                            }
                            __syncthreads();
                            if ((grp >> lane) & 1u) lns = sm.bn[lane].ns;
                        }
                        nr = 0;
                        for (unsigned m = grp; m; m &= m - 1) {
                            const int bi = __ffs(m) - 1, ns = __shfl_sync(0xffffffffu, lns, bi);
                            if (bi % NWARPS == warp) lay_out(sm.bn[bi], nr, 0, ns, false);
                            nr += ns;
                        }
                        pre = false;
                        suf = true;
                        continue;
                    }
                    for (unsigned m = grp; m; m &= m - 1) {
                        const int bi = __ffs(m) - 1;
                        if (bi % NWARPS == warp) decide_open(sm.bn[bi], dout);
                    }
                }
                if (!left) {
                    __syncthreads();
                    break;
                }
                // the next open nodes
                const unsigned dm = __ballot_sync(0xffffffffu, ((left >> lane) & 1u) && sm.bn[lane].direct);
                int np = 0, ns = 0;
                grp = 0u;
                dir = true;
                while (left) {
                    const int bi = __ffs(left) - 1;
                    const int p = __shfl_sync(0xffffffffu, lnp, bi), q = __shfl_sync(0xffffffffu, lns, bi);
                    const bool d = dir && ((dm >> bi) & 1u);
                    if (grp && (np + p > kNCR || ns + q > kNCR)) break;   // (a node's own always fit)
                    // with a direction on each half of the warps, both at once while they fit
                    if (DIRS == 2 && grp && np + ns + p + q > (d ? A.nrow : kNCR)) break;
                    np += p;
                    ns += q;
                    dir = d;
                    grp |= 1u << bi;
                    left &= left - 1;
                }
                suf = np + ns <= kNCR || (dir && np + ns <= A.nrow);
                pre = true;
                dout = suf ? 0 : S::NROW;
                nr = 0;
                for (unsigned m = grp; m; m &= m - 1) {
                    const int bi = __ffs(m) - 1;
                    const int p = __shfl_sync(0xffffffffu, lnp, bi), q = suf ? __shfl_sync(0xffffffffu, lns, bi) : 0;
                    if (bi % NWARPS == warp) lay_out(sm.bn[bi], nr, p, q, true);
                    nr += p + q;
                }
            }
            // ---- phase D2: numbering, children, gains, keys (warp per node) --------
            // Child indices are deterministic: the batch's nodes in order, after the
            // nodes created before this batch.
            for (int bi = warp; bi < nb; bi += NWARPS) {
                const BatchNode &B = sm.bn[bi];
                NodeS &nd = sm.nodes[B.node];
                const int64_t gv = gidx(B.node);
                int before = lane < bi ? max((int)sm.bn[lane].nchild, 0) : 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
                const int nch = B.nchild;
                if (nch < 0) {   // pending root
                    if (lane == 0) {
                        const float bnd = B.forced ? FLT_MAX : split_bound(nd.kin, sm.rootR, nd.D);
                        nd.nchild = -1;
                        A.nd_child0[gv] = -1; A.nd_nchild[gv] = -1; A.nd_cost[gv] = 0;
                        A.nd_U[gv] = bnd; A.nd_kappa[gv] = 0.f; A.nd_sel[gv] = 0;
                        atomicMax(reinterpret_cast<int *>(&sm.pend), __float_as_int(bnd));
                    }
                    continue;
                }
                const int child0 = nch ? nn + before : -1;
                if (nch == 0) {
                    if (lane == 0) {
                        nd.nchild = 0;
                        A.nd_child0[gv] = -1; A.nd_nchild[gv] = 0; A.nd_cost[gv] = 0;
                        A.nd_U[gv] = 0.f; A.nd_kappa[gv] = 0.f; A.nd_sel[gv] = 0;
                    }
                    continue;
                }
                float rch[3] = {0.f, 0.f, 0.f};
                for (int q = 0; q < nch; q++) {
                    float r = 0.f;
                    for (int t = B.ca[q] + lane; t < B.cb[q]; t += 32) r += sm.RK[t].x;
                    rch[q] = warp_sum(r);
                }
                const float rnode = (rch[0] + rch[1]) + rch[2];   // R of the node = sum over its children
                const float dsum = (B.cD[0] + B.cD[1]) + (nch == 3 ? B.cD[2] : 0.f);
                const int cost = nch - 1;
                float gain = om * rnode * (nd.D - dsum);
                if (gain < 0.f) gain = 0.f;
                const float U = cost == 2 ? 0.5f * gain : gain;
                const float kap = B.forced ? FLT_MAX : fminf(U, nd.kin);
                if (lane == 0) {
                    nd.nchild = (signed char)nch;
                    A.nd_child0[gv] = (int32_t)(gidx(child0) - nbase); A.nd_nchild[gv] = (int8_t)nch;
                    A.nd_cost[gv] = (int8_t)cost; A.nd_U[gv] = U; A.nd_kappa[gv] = kap;
                    A.nd_sel[gv] = 0;
                    A.ops[sm.op_base + B.op] = make_uint2(__float_as_uint(kap), ((uint32_t)gv << 1) | (uint32_t)(cost - 1));
                }
                if (lane < nch) {   // lane q writes child q
                    const int q = lane, ci = child0 + q;
                    const float rq = q == 0 ? rch[0] : (q == 1 ? rch[1] : rch[2]);
                    NodeS &ch = sm.nodes[ci];
                    ch.a = B.ca[q]; ch.b = B.cb[q]; ch.nchild = 0; ch.D = B.cD[q]; ch.kin = kap;
                    const int64_t gc = gidx(ci);
                    A.nd_a[gc] = sa + B.ca[q]; A.nd_b[gc] = sa + B.cb[q];
                    A.nd_parent[gc] = (int32_t)gv; A.nd_unit[gc] = (int32_t)uid;
                    A.nd_D[gc] = B.cD[q]; A.nd_R[gc] = (float)rq;
                    A.nd_child0[gc] = -1; A.nd_nchild[gc] = 0; A.nd_cost[gc] = 0;
                    // until the child is evaluated, nd_U holds the bound of its split key
                    // (the largest key when it holds a floor position: a floor op)
                    bool chf = false;
                    if (ufl)
                        for (int t = B.ca[q]; t < B.cb[q] && !chf; t++) chf = sm.Ff[t] > -INFINITY;
                    const float cbnd = B.cb[q] - B.ca[q] >= 2 ? (chf ? FLT_MAX : split_bound(kap, rq, B.cD[q])) : 0.f;
                    A.nd_U[gc] = cbnd;
                    A.nd_kappa[gc] = 0.f; A.nd_sel[gc] = 0;
                    if (B.cb[q] - B.ca[q] >= 2) {
                        if (cbnd >= A.tau && levels_left > 0) {   // evaluated at the next level of this launch
                            atomicOr(&sm.lvl[cur ^ 1][ci >> 5], 1u << (ci & 31));
                        } else {   // the launch's last level, or a key that cannot reach its threshold
                            ch.nchild = -1;
                            A.nd_nchild[gc] = -1;
                            atomicMax(reinterpret_cast<int *>(&sm.pend), __float_as_int(cbnd));
                        }
                    }
                }
            }
            // nodes created by this batch
            nn += __reduce_add_sync(0xffffffffu, lane < nb ? max((int)sm.bn[lane].nchild, 0) : 0);
            __syncthreads();
        }
    }
    if (lane == 0) { sm.wcnt[warp][0] = w_scan; sm.wcnt[warp][1] = w_eval; sm.wcnt[warp][2] = w_len; }
    __syncthreads();
    if (tid == 0) {
        if constexpr (!SUB) {   // a subtree stays inside its reserved slots; what it left pending is never needed
            A.u_nnodes[uid] = nn;
            A.u_pend[uid] = sm.pend;
        }
        if (fresh) A.u_sel[uid] = 0;
        unsigned long long tot[3] = {0, 0, 0};
        for (int w = 0; w < NWARPS; w++)
            for (int q = 0; q < 3; q++) tot[q] += sm.wcnt[w][q];
        atomicAdd(&A.work[0], tot[0]);
        atomicAdd(&A.work[1], tot[1]);
        atomicAdd(&A.work[2], tot[2]);
        atomicAdd(&A.work[3], 1ull);
    }
    // unused node slots of the unit carry cost 0 (no op)
    if (fresh)
        for (int k = nn + tid; k < 2 * n; k += NT) A.nd_cost[nbase + k] = 0;
}

template <int DH, typename Tin, int NMAX, bool SUB = false>
cudaError_t launch_t(Ctx &c, BuildArgs &A, unsigned grid, cudaStream_t s) {
    using S = Smem<DH, NMAX>;
    static_assert(sizeof(S) <= 227 * 1024, "unit kernel shared memory above the per-CTA limit");
    static_assert((sizeof(S) + 1024) * S::CTAS <= 228 * 1024, "unit kernel shared memory above the SM's");
    if (grid == 0) return cudaSuccess;
    // rows for both sides of a node only where nodes evaluate all cuts at once:
    // the L1 cache keeps the rest
    A.nrow = A.prune && A.lam_kappa >= kDirectMax ? kNCR : S::NROW;
    const size_t sm = sizeof(S) - (S::NROW - A.nrow) * S::ROWF * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(unit_build_kernel<DH, Tin, NMAX, SUB>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(S));
    if (e != cudaSuccess) return e;
    unit_build_kernel<DH, Tin, NMAX, SUB><<<grid, S::NT, sm, s>>>(A);
    c.launches += 1;
    return cudaGetLastError();
}

template <typename Tin, int NMAX, bool SUB = false>
cudaError_t launch_dt(Ctx &c, BuildArgs &A, unsigned grid, cudaStream_t s) {
    return c.p.d == 128 ? launch_t<128, Tin, NMAX, SUB>(c, A, grid, s) : launch_t<64, Tin, NMAX, SUB>(c, A, grid, s);
}

}  // namespace

static void fill_args(BuildArgs &A, Ctx &c, const void *K, const void *V, const void *Q, const float *omega,
                      const int32_t *slots, int J) {
    const gkv_params &p = c.p;
    A.K = K; A.V = V; A.Q = Q;
    A.slots = slots; A.rope = c.w.rope; A.kappa = c.w.kappa;
    A.rtok = c.w.rtok; A.row_m = c.w.row_m; A.row_Z = c.w.row_Z; A.omega = omega;
    A.Eg = use_tc(c) ? c.w.Eg : nullptr;   // written by the tensor-core pass B
    A.fl_acc = p.alpha_floor > 0.0 ? c.w.fl_acc : nullptr;
    A.fl_f = c.w.fl_f;
    A.L = p.L; A.G = p.G; A.Hq = p.Hq; A.T = p.T; A.d = p.d; A.W = p.W; A.gq = p.Hq / p.G;
    A.cs = p.ctx_start; A.Nc = c.Nc; A.J = J; A.k_cand = p.k_cand;
    A.inv_sqrt_d = (float)(1.0 / sqrt((double)p.d));
    A.lamZ = (float)p.lambda_Z; A.lamM = (float)p.lambda_M; A.eps = (float)p.eps;
    A.lam_kappa = p.lambda_kappa; A.base_frac = p.base_frac;
    A.prune = p.lambda_Z >= 0.0 && p.lambda_M >= 0.0;
    A.nd_a = c.w.nd_a; A.nd_b = c.w.nd_b; A.nd_child0 = c.w.nd_child0;
    A.nd_parent = c.w.nd_parent; A.nd_unit = c.w.nd_unit;
    A.nd_nchild = c.w.nd_nchild; A.nd_cost = c.w.nd_cost;
    A.ops = c.w.ops; A.n_ops = c.w.n_ops;
    A.nd_D = c.w.nd_D; A.nd_R = c.w.nd_R; A.nd_U = c.w.nd_U; A.nd_kappa = c.w.nd_kappa;
    A.nd_sel = c.w.nd_sel;
    A.u_nnodes = c.w.u_nnodes; A.u_Uadd = c.w.u_Uadd; A.u_Ddrop = c.w.u_Ddrop; A.u_sel = c.w.u_sel;
    A.u_pend = c.w.u_pend;
    A.status = c.w.dev_int + 1;
    A.work = c.w.work;
}

// One launch per class, `per` CTAs per listed item.  Classes that together fit
// one wave of a larger instance's CTAs share its launch.
template <typename Tin, bool SUB>
static cudaError_t launch_classes(Ctx &c, BuildArgs &A, const UnitLists &u, unsigned per, cudaStream_t s) {
    const int64_t n0 = (int64_t)u.cnt[0] * per, n1 = (int64_t)u.cnt[1] * per, n2 = (int64_t)u.cnt[2] * per;
    const int far = 1 << 30;
    A.stride = u.stride;
    auto range = [&](int a, int b) {   // classes [a, b]: returns the CTAs
        A.list = u.list + a * u.stride;
        A.c1 = b > a ? u.cnt[a] : far;
        A.c2 = b > a + 1 ? u.cnt[a] + u.cnt[a + 1] : far;
        int64_t n = 0;
        for (int q = a; q <= b; q++) n += (int64_t)u.cnt[q] * per;
        return (unsigned)n;
    };
    if (n0 + n1 + n2 <= c.num_sms) return launch_dt<Tin, kMaxUnit, SUB>(c, A, range(0, 2), s);
    cudaError_t e = cudaSuccess;
    if (n0 + n1 <= 2 * c.num_sms) {
        e = launch_dt<Tin, kShortUnit, SUB>(c, A, range(0, 1), s);
    } else {
        e = launch_dt<Tin, kTinyUnit, SUB>(c, A, range(0, 0), s);
        if (e == cudaSuccess) e = launch_dt<Tin, kShortUnit, SUB>(c, A, range(1, 1), s);
    }
    if (e == cudaSuccess) e = launch_dt<Tin, kMaxUnit, SUB>(c, A, range(2, 2), s);
    return e;
}

cudaError_t launch_unit_build(Ctx &c, const void *K, const void *V, const void *Q,
                              const float *omega, const int32_t *slots, int J, int resume,
                              int root_only, int max_levels, float tau, const UnitLists &u, cudaStream_t s,
                              int lg0, int nlg) {
    BuildArgs A;
    fill_args(A, c, K, V, Q, omega, slots, J);
    A.resume = resume; A.root_only = root_only; A.max_levels = max_levels; A.tau = tau;
    if (nlg < 0) nlg = c.p.L * c.p.G - lg0;
    A.lg0 = lg0;
    A.nlg = nlg;
    const unsigned per = resume ? 1u : (unsigned)nlg;
    return c.p.dtype == GKV_BF16 ? launch_classes<__nv_bfloat16, false>(c, A, u, per, s)
                                 : launch_classes<float, false>(c, A, u, per, s);
}

cudaError_t launch_unit_subtrees(Ctx &c, const void *K, const void *V, const void *Q, const float *omega,
                                 const int32_t *slots, int J, const UnitLists &u, float tau_prune,
                                 cudaStream_t s) {
    BuildArgs A;
    fill_args(A, c, K, V, Q, omega, slots, J);
    A.resume = 0; A.root_only = 0; A.max_levels = 4 * kMaxUnit; A.tau = tau_prune;
    A.lg0 = 0;
    A.nlg = c.p.L * c.p.G;
    return c.p.dtype == GKV_BF16 ? launch_classes<__nv_bfloat16, true>(c, A, u, 1, s)
                                 : launch_classes<float, true>(c, A, u, 1, s);
}

}  // namespace gkv
