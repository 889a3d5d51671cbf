// cc_mixed.cu -- mixed-precision forms of the two pair kernels of the CC
// split (arXiv:1407.7105, Eqs. tauij, kickij/kickji):
//
//  * k_tau_mixed: the edge predicate tau(i,j) < h decided in FP32 with a
//    rigorous per-pair error bound; a pair whose FP32 value is too close to
//    h for the bound to decide is re-evaluated with the exact FP64
//    predicate (tau_fp64), so the edge set is identical to the FP64 one.
//    Every split of both forms (and the OK split's outer level) runs it.
//  * k_kick_mixed: pair forces in FP32 from float-float position
//    differences, rsqrt plus one Newton step, Kahan-compensated FP32 sums,
//    partial sums over j-chunks combined in FP64; v stays FP64.
//
// Positions and velocities are carried as float pairs (hi = fl32(x),
// lo = fl32(x - hi)), so x_j - x_i = (hi_j - hi_i) + (lo_j - lo_i) is formed
// with relative error <= 2u + 11 u^2 X / r (u = 2^-24, X = max |x|),
// the accuracy of an FP64 difference rounded to FP32 up to one more
// rounding, at three FP32 additions instead of three FP64 subtractions
// (GB300 issues FP64 at 1/58 of the FP32 rate).
#include "cc_device.cuh"

namespace cc {

// ------------------------------------------------------------ prep
// float-float copy of the packed state; per-level maxima of |x| and |v|
__global__ void k_prep_ff(Level L, FFView F, float G, int with_v, int init_forest, unsigned long long *edge_count)
{
    pdl_begin();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    float ax = 0.f, av = 0.f;
    if (init_forest) {
        // the split's union-find starts as singletons (what k_init_parent does)
        if (k < L.total) {
            L.parent[k] = k;
            L.cnt[k] = 0;
        }
        if (k == 0 && edge_count) *edge_count = 0ull;
    }
    if (k < L.total && L.gid[k] >= 0) {
        const double xs[3] = {L.x[k], L.y[k], L.z[k]};
        float hi[3], lo[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            ff_split(xs[c], hi[c], lo[c]);
            ax = fmaxf(ax, fabsf(hi[c]));
        }
        F.pq[2 * k] = make_float4(hi[0], hi[1], hi[2], G * fl32(L.m[k]));
        F.pq[2 * k + 1] = make_float4(lo[0], lo[1], lo[2], 0.f);
        const float xh[3] = {hi[0], hi[1], hi[2]};
        if (with_v) {
            const double vs[3] = {L.vx[k], L.vy[k], L.vz[k]};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                ff_split(vs[c], hi[c], lo[c]);
                av = fmaxf(av, fabsf(hi[c]));
            }
            F.vq[2 * k] = make_float4(hi[0], hi[1], hi[2], 0.f);
            F.vq[2 * k + 1] = make_float4(lo[0], lo[1], lo[2], 0.f);
            float *h = reinterpret_cast<float *>(F.hp) + (size_t)(k >> 1) * 12 + (k & 1);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                h[2 * c] = xh[c];
                h[6 + 2 * c] = hi[c];
            }
        }
    }
    // positive floats order like their bit patterns
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ax = fmaxf(ax, __shfl_xor_sync(0xffffffffu, ax, o));
        av = fmaxf(av, __shfl_xor_sync(0xffffffffu, av, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (ax > 0.f) atomicMax((int *)&F.maxes[0], __float_as_int(ax));
        if (av > 0.f) atomicMax((int *)&F.maxes[1], __float_as_int(av));
    }
}

void launch_prep_ff(const Level &L, const FFView &F, double G, bool with_v, cudaStream_t s, bool init,
                    unsigned long long *edge_count)
{
    if (L.total <= 0) return;
    if (init) cudaMemsetAsync(F.maxes, 0, 2 * sizeof(float), s);
    launch_next(k_prep_ff, (L.total + 255) / 256, 256, 0, s, L, F, (float)G, with_v ? 1 : 0, init ? 1 : 0,
                                                    edge_count);
    CC_COUNT_LAUNCH(1);
}

// The packed kick's copy, in F.pq's place: two bodies together, four float4 a pair
//   (x x' y y') (z z' Gm Gm') (xlo xlo' ylo ylo') (zlo zlo' - -)
// so that the pair loop's packed operands come straight from a 16-byte load.
__device__ __forceinline__ float *kick_slot(const FFView &F, int t)
{
    return reinterpret_cast<float *>(F.pq) + (size_t)(t >> 1) * 16 + (t & 1);
}

// positions (hi, G m), (lo) and labels in the root-sorted order of the
// split: position t holds packed element order[t].  dt > 0: the level's
// first drift D_{h/2,T_R} of rest-set members (component size 1, Eq. drift,
// exact IEEE operations) is applied first, in the same pass.
__global__ void k_prep_kick(Level L, FFView F, const int32_t *order, const int32_t *root, float G, double dt,
                            int packed)
{
    pdl_begin();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= L.total) return;
    const int k = order[t];
    if (L.gid[k] < 0) {
        L.klab[t] = -1 - t;
        return;
    }
    if (dt > 0.0 && L.cnt[root[k]] == 1) {
        L.x[k] = __dadd_rn(L.x[k], __dmul_rn(dt, L.vx[k]));
        L.y[k] = __dadd_rn(L.y[k], __dmul_rn(dt, L.vy[k]));
        L.z[k] = __dadd_rn(L.z[k], __dmul_rn(dt, L.vz[k]));
    }
    const double xs[3] = {L.x[k], L.y[k], L.z[k]};
    float hi[3], lo[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) ff_split(xs[c], hi[c], lo[c]);
    const float gm = G * fl32(L.m[k]);
    if (!packed) {
        F.pq[2 * t] = make_float4(hi[0], hi[1], hi[2], gm);
        F.pq[2 * t + 1] = make_float4(lo[0], lo[1], lo[2], 0.f);
    } else {
        float *q = kick_slot(F, t);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            q[2 * c] = hi[c];
            q[8 + 2 * c] = lo[c];
        }
        q[6] = gm;
    }
    L.klab[t] = root[k];
}

void launch_prep_kick(const Level &L, const FFView &F, const int32_t *order, const int32_t *root, double G,
                      double drift_dt, bool packed, cudaStream_t s)
{
    if (L.total <= 0) return;
    launch_next(k_prep_kick, (L.total + 255) / 256, 256, 0, s, L, F, order, root, (float)G, drift_dt, packed ? 1 : 0);
    CC_COUNT_LAUNCH(1);
}

// ------------------------------------------------------------ tau
// One block per triangular tile (T x T pairs) of a set: each warp holds 32 R
// rows (R per lane) against T/S columns of the tile (S > 1 splits the
// columns over more warps, for sets with few tiles).
//
// What bounds it: the FP32 pipes.  The certificates are three comparisons a
// pair (tau_pair_bounds: no square root; 13 FP32 operations against ~35 and
// three reciprocal square roots for tau_quick_apart), formed for two columns
// at a time with the packed FP32 instructions (add/fma .f32x2: one issue slot
// for two pairs), so a pair costs ~10 issue slots (~12 in cold groups, whose speed
// bound is each pair's own: TAU_FAR); the comparisons' outcomes
// are the sign bits of two sums, shifted into a 32-column mask per lane, so
// there is no vote and no branch per column.  Pairs left open are queued per
// warp and settled 32 at a time by the certified decision.
// Measured (GB300): top level of the 16384-body Plummer sphere (1.34e8 pairs)
// 252 -> 126 us, 65536-body fractal (2.1e9 pairs) 1798 -> 807 us, 40009 bodies
// in no spatial order (8.0e8 pairs) 1790 -> 630 us, before -> after the
// comparisons took the place of tau_quick_apart.  In a spatial order the
// launch ends with the tiles on the diagonal, whose pairs are mostly edges:
// four warps a 128-wide tile (R = 1) instead of two took the 16384-body level
// from 196 to 126 us.
// RAW: the set is a caller's FP64 arrays (L.x .. L.m, L.total bodies, no
// float-float copy): columns and rows are rounded as they are loaded.
constexpr int TAU_JG = 8;  // columns per group of the group certificates
// The pairs' own speed bounds (tau_pair_far, TAU_FAR: three packed operations more
// for two pairs) from v_thr = span/16 on, the widest relative speed per component of
// the two groups: where v_thr leaves a few pairs in a hundred open, settling them
// takes longer than the better bound.  Measured, tau kernel, with v_thr alone / the
// column test of before it / now: 16384-body spheres at h = 1/1024, virial ratio 0.5
// 0.122 / 0.283 / 0.122 ms, 0.02 0.421 / 0.267 / 0.107, 0.01 0.794 / 0.267 / 0.105, 0.001
// 0.425 / 0.267 / 0.105; 40009 bodies, 0.005 4.64 / 1.51 / 0.48; 32768-body fractal with a
// mass spectrum, 0.3 0.755 / 1.021 / 0.352.  span/4 and span/8 were slower in all of
// these (0.173 and 0.109 at 0.02), span/32 and span/64 within 2 %, but for hot spheres
// (40009 bodies, 0.5: 0.49 and 0.52 against 0.48).
constexpr float TAU_FAR_SPAN = 1.f / 256.f;

template <int T, int S, int R>
struct __align__(16) MixedTauSmem {
    static constexpr int W = T * S / (32 * R);  // warps
    float4 hp[3 * T / 2];                       // high parts of the j-tile, two bodies together (FFView::hp)
    int32_t lp[2 * T];                          // local union-find over the tile's particles
    uint32_t q[W][64];                          // per warp: pairs waiting for the certified decision
    uint32_t ent[W][128];                       // per warp: edges waiting to be recorded, and their tau
    double tau[W][128];
    GroupBox jb[T / TAU_JG];                    // boxes of the j-tile's TAU_JG-column groups
    float4 gq[W][T / S / TAU_JG];               // per warp and column group: p0, w0, what to do (TauKind), mu
    float2 gf[W][T / S / TAU_JG];               // and a, k (TAU_FAR)
    uint64_t bar;
};

enum TauKind : int { TAU_BOUNDS = 0, TAU_SPEED = 1, TAU_OPEN = 2, TAU_FAR = 3 };

// min / max over each aligned segment of W lanes (a whole warp: one
// instruction)
template <int W>
__device__ __forceinline__ float warp_min(float v)
{
    if constexpr (W == 32) {
        asm volatile("redux.sync.min.f32 %0, %0, 0xffffffff;" : "+f"(v));
        return v;
    }
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <int W>
__device__ __forceinline__ float warp_max(float v)
{
    if constexpr (W == 32) {
        asm volatile("redux.sync.max.f32 %0, %0, 0xffffffff;" : "+f"(v));
        return v;
    }
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// widens box B to the boxes of all lanes of each aligned segment of W lanes
// (a lane without a body brings an empty box: +-inf, Gm = 0)
template <int W>
__device__ __forceinline__ void warp_group_box(GroupBox &B)
{
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        B.xlo[k] = warp_min<W>(B.xlo[k]);
        B.xhi[k] = warp_max<W>(B.xhi[k]);
        B.vlo[k] = warp_min<W>(B.vlo[k]);
        B.vhi[k] = warp_max<W>(B.vhi[k]);
        a = fmaxf(a, fmaxf(fabsf(B.xlo[k]), fabsf(B.xhi[k])));
        b = fmaxf(b, fmaxf(fabsf(B.vlo[k]), fabsf(B.vhi[k])));
    }
    B.gm = warp_max<W>(B.gm);
    B.amax = a;
    B.vabs = b;
}

__device__ __forceinline__ void box_empty(GroupBox &B)
{
    const float inf = __int_as_float(0x7f800000);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        B.xlo[k] = B.vlo[k] = inf;
        B.xhi[k] = B.vhi[k] = -inf;
    }
    B.gm = 0.f;
}

// adds one body to box B; returns whether it is outside what the bounds
// allow for (tau_in_box)
__device__ __forceinline__ bool box_add(GroupBox &B, const float s[6], float gm)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        B.xlo[k] = fminf(B.xlo[k], s[k]);
        B.xhi[k] = fmaxf(B.xhi[k], s[k]);
        B.vlo[k] = fminf(B.vlo[k], s[3 + k]);
        B.vhi[k] = fmaxf(B.vhi[k], s[3 + k]);
    }
    // (a negative mass, which only a caller's own arrays can hold, has no largest
    // mu: no test of the group then takes its pairs)
    B.gm = gm >= 0.f ? fmaxf(B.gm, gm) : CUDART_INF_F;
    return !tau_in_box(s, gm);
}

// local union-find in shared memory (indices 0..2T-1, links to the smaller)
__device__ __forceinline__ int luf_find(volatile int32_t *p, int x)
{
    while (true) {
        const int q = p[x];
        if (q == x) return x;
        const int g = p[q];
        if (g != q) p[x] = g;
        x = q;
    }
}

__device__ __forceinline__ bool luf_union(int32_t *p, int a, int b)
{
    volatile int32_t *vp = p;
    for (int it = 0; it < (1 << 20); ++it) {
        a = luf_find(vp, a);
        b = luf_find(vp, b);
        if (a == b) return true;
        if (a > b) {
            const int t = a; a = b; b = t;
        }
        if (atomicCAS(&p[b], b, a) == b) return true;
    }
    return false;
}

// the high parts of body k and its G m
template <bool RAW>
__device__ __forceinline__ void tau_load_hi(const Level &L, const FFView &F, const MixedTauParams &Q, int k,
                                            float s[6], float &gm)
{
    if constexpr (RAW) {
        s[0] = fl32(L.x[k]); s[1] = fl32(L.y[k]); s[2] = fl32(L.z[k]);
        s[3] = fl32(L.vx[k]); s[4] = fl32(L.vy[k]); s[5] = fl32(L.vz[k]);
        gm = Q.G * fl32(L.m[k]);
    } else {
        const float4 p = F.pq[2 * k], v = F.vq[2 * k];
        s[0] = p.x; s[1] = p.y; s[2] = p.z;
        s[3] = v.x; s[4] = v.y; s[5] = v.z;
        gm = p.w;
    }
}

// the certified decision of one pair from its float-float differences; OWN: in
// units of the pair's own
template <bool RAW, bool OWN>
__device__ __forceinline__ int tau_decide_pair(const Level &L, const FFView &F, const MixedTauParams &Q, int i, int j)
{
    constexpr float c11 = 11.f * U32 * U32;
    float d[6], mu, cx, cv;
    if constexpr (RAW) {
        const double *src[6] = {L.x, L.y, L.z, L.vx, L.vy, L.vz};
        float big[2] = {0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            float ih, il, jh, jl;
            ff_split(src[c][i], ih, il);
            ff_split(src[c][j], jh, jl);
            d[c] = (jh - ih) + (jl - il);
            big[c / 3] = fmaxf(big[c / 3], fmaxf(fabsf(ih), fabsf(jh)));
        }
        // (with a negative mass the sum can cancel, and has no relative error bound)
        const float gi = Q.G * fl32(L.m[i]), gj = Q.G * fl32(L.m[j]);
        mu = gi >= 0.f && gj >= 0.f ? gi + gj : CUDART_NAN_F;
        cx = c11 * big[0];
        cv = c11 * big[1];
    } else {
        const float4 a0 = F.pq[2 * i], a1 = F.pq[2 * i + 1], b0 = F.vq[2 * i], b1 = F.vq[2 * i + 1];
        const float4 p0 = F.pq[2 * j], p1 = F.pq[2 * j + 1], v0 = F.vq[2 * j], v1 = F.vq[2 * j + 1];
        d[0] = (p0.x - a0.x) + (p1.x - a1.x);
        d[1] = (p0.y - a0.y) + (p1.y - a1.y);
        d[2] = (p0.z - a0.z) + (p1.z - a1.z);
        d[3] = (v0.x - b0.x) + (v1.x - b1.x);
        d[4] = (v0.y - b0.y) + (v1.y - b1.y);
        d[5] = (v0.z - b0.z) + (v1.z - b1.z);
        mu = a0.w + p0.w;
        cx = c11 * F.maxes[0];
        cv = c11 * F.maxes[1];
    }
    if constexpr (OWN) return tau_decide_own(d, mu, cx, cv, Q);
    else return tau_decide_at(tau_prep_fp32(d[0], d[1], d[2], d[3], d[4], d[5], mu, cx, cv, Q), Q.etah);
}

// an edge of each lane with `edge`: the local union, and a place in the warp's list
// of edges to record (ne of them so far); returns those lanes
template <int T, int S, int R>
__device__ __forceinline__ unsigned tau_edges(MixedTauSmem<T, S, R> &sm, int w, bool edge, unsigned ent, double tau,
                                              int ne, int joff, DevCounters *ctr, const EdgeList &E)
{
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    const unsigned eb = __ballot_sync(0xffffffffu, edge);
    if (edge && !luf_union(sm.lp, (int)(ent >> 8), joff + (int)(ent & 255u))) raise_err(ctr, DERR_UF_RETRY);
    if (edge && E.rec) {
        const int q = ne + __popc(eb & lt);
        sm.ent[w][q] = ent;
        sm.tau[w][q] = tau;
    }
    return eb;
}

// Settles the warp's queued pairs sm.q[w][0..cnt), one per lane, by the certified
// FP32 decision on the float-float differences.  Out of line: the pair loop
// keeps only the high parts and its masks in registers.  Returns (lanes whose
// pair is an edge, lanes whose pair is undecided: for tau_settle_open).
template <int T, int S, int R, bool RAW>
__device__ __noinline__ uint2 tau_settle_batch(MixedTauSmem<T, S, R> &sm, int w, int cnt, int ne, int ibase, int j0,
                                               int joff, const Level &L, const FFView &F, const MixedTauParams &Q,
                                               DevCounters *ctr, const EdgeList &E)
{
    const int lane = threadIdx.x & 31;
    const bool has = lane < cnt;
    const unsigned ent = has ? sm.q[w][lane] : 0u;
    int dec = 0;
    // (RAW: the float pairs again in the open batch would spill)
    if (has) dec = tau_decide_pair<RAW, RAW>(L, F, Q, ibase + (int)(ent >> 8), j0 + (int)(ent & 255u));
    const unsigned ub = __ballot_sync(0xffffffffu, dec < 0);
    return make_uint2(tau_edges(sm, w, dec > 0, ent, CUDART_NAN, ne, joff, ctr, E), ub);
}

// The undecided ones of them (lanes ub): the decision in the pair's own units (in
// units far from 1 the batch above leaves every pair open), else the exact FP64
// predicate (logged when near the threshold).  Returns (lanes whose pair is an
// edge, FP64 evaluations of this lane's pair).  Apart from the batch above, which
// is the common one: own units for all of its pairs took 3 % of a level by the unit
// calls (40009 bodies, 1.73 against 1.67 ms).
template <int T, int S, int R, bool RAW>
__device__ __noinline__ uint2 tau_settle_open(MixedTauSmem<T, S, R> &sm, int w, unsigned ub, int ne, int ibase, int j0,
                                              int joff, const Level &L, const FFView &F, const TauParams &P,
                                              const MixedTauParams &Q, DevCounters *ctr, int32_t *near_ij,
                                              double *near_tau, long long near_cap, const EdgeList &E)
{
    const int lane = threadIdx.x & 31;
    const unsigned ent = (ub >> lane) & 1u ? sm.q[w][lane] : 0u;
    bool edge = false;
    unsigned nfp64 = 0u;
    double tau = CUDART_NAN;
    if ((ub >> lane) & 1u) {
        const int gi = ibase + (int)(ent >> 8), gj = j0 + (int)(ent & 255u);
        int dec = -1;
        if constexpr (!RAW) dec = tau_decide_pair<false, true>(L, F, Q, gi, gj);
        edge = dec > 0;
        if (dec < 0) {
            tau = tau_fp64(__dsub_rn(L.x[gi], L.x[gj]), __dsub_rn(L.y[gi], L.y[gj]), __dsub_rn(L.z[gi], L.z[gj]),
                           __dsub_rn(L.vx[gi], L.vx[gj]), __dsub_rn(L.vy[gi], L.vy[gj]), __dsub_rn(L.vz[gi], L.vz[gj]),
                           L.m[gi], L.m[gj], P);
            nfp64 = 1u;
            if (fabs(tau - P.h) < P.near_tol * P.h) {
                const unsigned long long q = atomicAdd(&ctr->near_pairs, 1ull);
                if ((long long)q < near_cap) {
                    const int pi = L.gid[gi], pj = L.gid[gj];
                    near_ij[2 * q] = pi < pj ? pi : pj;
                    near_ij[2 * q + 1] = pi < pj ? pj : pi;
                    near_tau[q] = tau;
                }
            }
            edge = tau < P.h;
        }
    }
    return make_uint2(tau_edges(sm, w, edge, ent, tau, ne, joff, ctr, E), nfp64);
}

// Records the warp's ne listed edges (the decision at h/2 is left to the first
// half's pass; tau = the FP64 value or NaN).  One counter update for up to
// 128 of them: its round trip to L2 is longer than settling a batch, and in a
// spatial order the tiles on the diagonal hold thousands of edges each.
template <int T, int S, int R>
__device__ __noinline__ void tau_record(MixedTauSmem<T, S, R> &sm, int w, int ne, int ibase, int j0, const EdgeList &E)
{
    const int lane = threadIdx.x & 31;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(E.count, (unsigned long long)ne);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int k = lane; k < ne; k += 32) {
        const unsigned long long q = base + (unsigned)k;
        if ((long long)q >= E.cap) break;
        const unsigned ent = sm.ent[w][k];
        EdgeRec r;
        r.a = ibase + (int)(ent >> 8);
        r.b = j0 + (int)(ent & 255u);
        r.e = -1;
        r.pad = 0;
        r.tau = sm.tau[w][k];
        E.rec[q] = r;
    }
}

// Parameters are grid constants: the out-of-line settle takes them by
// reference without a copy.
template <int T, int S, int R, bool RAW>
__global__ void __launch_bounds__(T *S / R, 768 * R / (T * S))
    k_tau_mixed(const __grid_constant__ Level L, const __grid_constant__ FFView F,
                const __grid_constant__ TauParams P, const __grid_constant__ MixedTauBounds Q, DevCounters *ctr,
                int32_t *near_ij, double *near_tau, long long near_cap, const __grid_constant__ EdgeList E)
{
    pdl_begin();
    constexpr int THREADS = T * S / R, NW = THREADS / 32, RW = T / (32 * R);
    constexpr int TC = T / S, GW = TC / TAU_JG;  // a warp's columns and column groups
    static_assert(T % (32 * R) == 0 && TC % 32 == 0 && T <= 256, "tile shape");
    __shared__ MixedTauSmem<T, S, R> sm;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, slice = w / RW;
    const int row0 = (w % RW) * 32 * R + lane;  // the lane's rows: row0 + 32 r
    int s = 0, t = blockIdx.x, n, start;
    if constexpr (RAW) {
        n = L.total;
        start = 0;
    } else {
        int lo = 0, hi = L.nsets;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (L.tile_off[mid] <= (int)blockIdx.x) lo = mid; else hi = mid;
        }
        s = lo;
        t -= L.tile_off[s];
        n = L.set_n[s];
        start = L.set_start[s];
    }
    // tile t of the set: by diagonals, the main one first.  In a spatial order
    // the edges lie near it, and a tile full of edges takes many times an
    // empty one's time: started last it would be the launch's tail.
    const int nt = (n + T - 1) / T;
    const int dt = tri_tile_row(t, nt);
    const int ti = t, tj = t + dt;
    const bool diag = dt == 0;
    const int ibase = start + ti * T, j0 = start + tj * T;
    const int ni = min(T, n - ti * T), jn = min(T, n - tj * T);
    for (int e = tid; e < 2 * T; e += THREADS) sm.lp[e] = e;
    if constexpr (RAW) {
        for (int p = tid; 2 * p < jn; p += THREADS) {
            float a[6], b[6], g;
            tau_load_hi<true>(L, F, Q, j0 + 2 * p, a, g);
            tau_load_hi<true>(L, F, Q, j0 + min(2 * p + 1, jn - 1), b, g);
#pragma unroll
            for (int c = 0; c < 3; ++c) sm.hp[3 * p + c] = make_float4(a[2 * c], b[2 * c], a[2 * c + 1], b[2 * c + 1]);
        }
        __syncthreads();
    } else {
        if (tid == 0) {
            mbar_init(&sm.bar, 1);
            fence_mbar_init();
        }
        __syncthreads();
        // fault_test = 1: the copy is announced but never issued, so the wait
        // below runs out (a test of the bounded wait; no copy is in flight)
        const bool no_copy = P.fault_test == 1;
        const long long wait_cycles = no_copy ? FAULT_TEST_WAIT_CYCLES : TMA_WAIT_CYCLES;
        if (tid == 0) {
            // (an odd last body brings its neighbour's slot along: masked below)
            const unsigned bytes = (unsigned)((jn + 1) / 2) * 48u;
            mbar_expect_tx(&sm.bar, bytes);
            if (!no_copy) tma_load_1d(sm.hp, F.hp + 3 * (size_t)(j0 / 2), bytes, &sm.bar);
        }
        const bool got = mbar_wait(&sm.bar, 0, wait_cycles);
        if (__syncthreads_or(!got)) {
            raise_err(ctr, DERR_TMA_TIMEOUT);
            // let a copy still in flight land before the CTA exits
            mbar_wait(&sm.bar, 0, wait_cycles);
            return;
        }
    }
    unsigned long long my_edges = 0, my_fp64 = 0;
    const int joff = diag ? 0 : T;  // local index base of the j-tile
    const unsigned lt = (1u << lane) - 1u;
    // ---- boxes: the column groups' (32 columns a round and warp), the rows'
    for (int c0 = 32 * w; c0 < T; c0 += 32 * NW) {
        const int k = c0 + lane;
        GroupBox B;
        box_empty(B);
        bool wild = false;
        if (k < jn) {
            const float *h = reinterpret_cast<const float *>(sm.hp) + (k >> 1) * 12 + (k & 1);
            const float st[6] = {h[0], h[2], h[4], h[6], h[8], h[10]};
            float gm;
            if constexpr (RAW) gm = Q.G * fl32(L.m[j0 + k]);
            else gm = F.pq[2 * (size_t)(j0 + k)].w;
            wild = box_add(B, st, gm);
        }
        warp_group_box<TAU_JG>(B);
        const unsigned wb = __ballot_sync(0xffffffffu, wild) >> (lane & ~(TAU_JG - 1));
        if ((lane & (TAU_JG - 1)) == 0) {
            if (k >= jn) B.gm = -1.f;                          // no bodies
            if (wb & ((1u << TAU_JG) - 1u)) B.gm = CUDART_INF_F;  // a body outside the bounds' range
            sm.jb[k / TAU_JG] = B;
        }
    }
    uint64_t nx[R][6];  // minus the row's high parts, twice each
    GroupBox A;
    box_empty(A);
    bool awild = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int row = row0 + 32 * r;
        float st[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, gm;
        if (row < ni) {
            tau_load_hi<RAW>(L, F, Q, ibase + row, st, gm);
            awild = box_add(A, st, gm) || awild;
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) nx[r][c] = pack2(-st[c], -st[c]);
    }
    warp_group_box<32>(A);
    awild = __any_sync(0xffffffffu, awild);
    __syncthreads();
    // ---- certificates of the warp's rows against each of its column groups
    if (lane < GW) {
        const GroupBox &B = sm.jb[slice * GW + lane];
        float4 g = make_float4(0.f, 0.f, __int_as_float(TAU_OPEN), A.gm + B.gm);
        if (!awild && B.gm >= 0.f && B.gm < CUDART_INF_F) {
            float thr;
            PairBounds b;
            if (!diag && tau_groups_apart(A, B, Q, thr)) {
                g.y = -thr;
                g.z = __int_as_float(TAU_SPEED);
            } else if (tau_pair_bounds(A.amax, A.vabs, A.gm + B.gm, Q, b)) {
                g.x = b.p0;
                g.y = b.w0;
                g.z = __int_as_float(TAU_BOUNDS);
                // v_thr beside the groups' speeds
                const float span = tau_speed_span(A, B);
                PairFar f;
                if (TAU_FAR_SPAN * span * span < -b.w0 &&
                    tau_pair_far(A.amax, A.vabs, fmaxf(A.amax, B.amax), span, A.gm + B.gm, Q, f)) {
                    g.x = f.p0;
                    g.y = f.w0;
                    g.z = __int_as_float(TAU_FAR);
                    sm.gf[w][lane] = make_float2(f.a, f.k);
                }
            }
        }
        sm.gq[w][lane] = g;
    }
    __syncwarp();
    const uint64_t nc2 = pack2(-Q.pb_c2, -Q.pb_c2);
    int qn = 0, ne = 0;  // pairs queued, edges listed by this warp (warp-uniform)
    auto listed = [&](unsigned eb) {  // edges just listed: counted, recorded when there are many
        const int k = __popc(eb);
        my_edges += lane == 0 ? k : 0;
        if (!E.rec) return;
        ne += k;
        __syncwarp();
        if (ne > 96) {
            tau_record<T, S, R>(sm, w, ne, ibase, j0, E);
            __syncwarp();
            ne = 0;
        }
    };
    auto settle = [&](int cnt) {
        const uint2 c = tau_settle_batch<T, S, R, RAW>(sm, w, cnt, ne, ibase, j0, joff, L, F, Q, ctr, E);
        listed(c.x);
        if (c.y != 0u) {
            const uint2 d = tau_settle_open<T, S, R, RAW>(sm, w, c.y, ne, ibase, j0, joff, L, F, P, Q, ctr, near_ij,
                                                          near_tau, near_cap, E);
            my_fp64 += d.y;
            listed(d.x);
        }
    };
    const int kb = slice * TC, k1 = min(jn, kb + TC);
#pragma unroll 1
    for (int cb = kb; cb < k1; cb += 32) {
        // columns cb..cb+31: bit 31 - c of m[r] = pair (row r, column cb + c) is open
        uint32_t m[R];
#pragma unroll
        for (int r = 0; r < R; ++r) m[r] = 0u;
        const int ng = min(4, (k1 - cb + TAU_JG - 1) / TAU_JG);
#pragma unroll 1
        for (int g = 0; g < ng; ++g) {
            const float4 gc = sm.gq[w][(cb - kb) / TAU_JG + g];
            const int kind = __float_as_int(gc.z);
            const ulonglong2 *J = reinterpret_cast<const ulonglong2 *>(sm.hp) + 3 * ((cb + TAU_JG * g) >> 1);
            if (kind == TAU_BOUNDS) {
                const uint64_t p0 = pack2(gc.x, gc.x), w0 = pack2(gc.y, gc.y);
#pragma unroll
                for (int u = 0; u < TAU_JG / 2; ++u) {
                    const ulonglong2 a = J[3 * u], b = J[3 * u + 1], c = J[3 * u + 2];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const uint64_t dx = add2(a.x, nx[r][0]), dy = add2(a.y, nx[r][1]), dz = add2(b.x, nx[r][2]);
                        const uint64_t du = add2(b.y, nx[r][3]), dv = add2(c.x, nx[r][4]), dw = add2(c.y, nx[r][5]);
                        const uint64_t oo = tau_pair_open(dx, dy, dz, du, dv, dw, p0, w0, nc2);
                        m[r] = __funnelshift_l((uint32_t)oo, m[r], 1);
                        m[r] = __funnelshift_l((uint32_t)(oo >> 32), m[r], 1);
                    }
                }
            } else if (kind == TAU_FAR) {
                const float2 gf = sm.gf[w][(cb - kb) / TAU_JG + g];
                const uint64_t p0 = pack2(gc.x, gc.x), w0 = pack2(gc.y, gc.y), fa = pack2(gf.x, gf.x), fk = pack2(gf.y, gf.y);
#pragma unroll
                for (int u = 0; u < TAU_JG / 2; ++u) {
                    const ulonglong2 a = J[3 * u], b = J[3 * u + 1], c = J[3 * u + 2];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const uint64_t dx = add2(a.x, nx[r][0]), dy = add2(a.y, nx[r][1]), dz = add2(b.x, nx[r][2]);
                        const uint64_t du = add2(b.y, nx[r][3]), dv = add2(c.x, nx[r][4]), dw = add2(c.y, nx[r][5]);
                        const uint64_t oo = tau_far_open(dx, dy, dz, du, dv, dw, p0, w0, nc2, fa, fk);
                        m[r] = __funnelshift_l((uint32_t)oo, m[r], 1);
                        m[r] = __funnelshift_l((uint32_t)(oo >> 32), m[r], 1);
                    }
                }
            } else if (kind == TAU_SPEED) {
                const uint64_t w0 = pack2(gc.y, gc.y);
#pragma unroll
                for (int u = 0; u < TAU_JG / 2; ++u) {
                    const uint64_t b = J[3 * u + 1].y;
                    const ulonglong2 c = J[3 * u + 2];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const uint64_t du = add2(b, nx[r][3]), dv = add2(c.x, nx[r][4]), dw = add2(c.y, nx[r][5]);
                        const uint64_t ww = tau_speed_open(du, dv, dw, w0);
                        m[r] = __funnelshift_l((uint32_t)ww, m[r], 1);
                        m[r] = __funnelshift_l((uint32_t)(ww >> 32), m[r], 1);
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) m[r] = (m[r] << TAU_JG) | ((1u << TAU_JG) - 1u);
            }
        }
        // the columns that exist, and (diagonal tiles) lie right of the row
        int open = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int row = row0 + 32 * r, c0 = diag ? max(0, row + 1 - cb) : 0, c1 = min(32, k1 - cb);
            m[r] <<= 32 - TAU_JG * ng;
            m[r] &= row < ni && c0 < c1 ? (0xffffffffu >> c0) & (0xffffffffu << (32 - c1)) : 0u;
            open += __popc(m[r]);
        }
        if (!__any_sync(0xffffffffu, open != 0)) continue;
        if (__reduce_add_sync(0xffffffffu, (unsigned)open) > 32u * 32u * R / 2u) {
            // most pairs open (groups outside the bounds' range): the full
            // certificate column by column is cheaper than settling them all.
            // (From a quarter, an eighth or a sixteenth of the pairs on it is
            // wasted where they are edges: 16384 bodies, h = 1/64, 1.03 -> 1.20-1.23 ms)
            for (int c = 0; c < min(32, k1 - cb); ++c) {
                const int k = cb + c;
                const float *h = reinterpret_cast<const float *>(sm.hp) + (k >> 1) * 12 + (k & 1);
                const float mu = sm.gq[w][(k - kb) / TAU_JG].w;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float d[6], x[6], e;
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        unpack2(nx[r][q], x[q], e);
                        d[q] = h[2 * q] + x[q];
                    }
                    const float cX = 7.1f * U32 * fmaxf(fabsf(x[0]), fmaxf(fabsf(x[1]), fabsf(x[2])));
                    const float cV = 7.1f * U32 * fmaxf(fabsf(x[3]), fmaxf(fabsf(x[4]), fabsf(x[5])));
                    if (tau_quick_apart(d[0], d[1], d[2], d[3], d[4], d[5], mu, cX, cV, Q)) m[r] &= ~(0x80000000u >> c);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            for (;;) {
                const unsigned b = __ballot_sync(0xffffffffu, m[r] != 0u);
                if (b == 0u) break;
                if (m[r] != 0u) {
                    const int c = __clz(m[r]);
                    m[r] &= ~(0x80000000u >> c);
                    sm.q[w][qn + __popc(b & lt)] = ((unsigned)(row0 + 32 * r) << 8) | (unsigned)(cb + c);
                }
                qn += __popc(b);
                if (qn >= 32) {
                    __syncwarp();
                    settle(32);
                    __syncwarp();
                    const uint32_t keep = lane < qn - 32 ? sm.q[w][32 + lane] : 0u;
                    __syncwarp();
                    if (lane < qn - 32) sm.q[w][lane] = keep;
                    qn -= 32;
                }
            }
        }
    }
    if (qn > 0) {
        __syncwarp();
        settle(qn);
    }
    if (ne > 0) tau_record<T, S, R>(sm, w, ne, ibase, j0, E);
    __syncthreads();
    // merge the tile's local components into the global forest: one union
    // per local non-root element instead of one per edge
    for (int e = tid; e < (diag ? T : 2 * T); e += THREADS) {
        const int r = luf_find(sm.lp, e);
        if (r != e) {
            const int ge = (e < T) ? ibase + e : j0 + (e - T);
            const int gr = (r < T) ? ibase + r : j0 + (r - T);
            // (fault_test = 2: every hook gives up at once, a test of the retry cap)
            if (!uf_union(L.parent, ge, gr, P.fault_test == 2 ? 0 : UF_RETRY_MAX)) raise_err(ctr, DERR_UF_RETRY);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_edges += __shfl_down_sync(0xffffffffu, my_edges, o);
        my_fp64 += __shfl_down_sync(0xffffffffu, my_fp64, o);
    }
    if ((tid & 31) == 0) {
        if (my_edges) atomicAdd(&ctr->edges, my_edges);
        if (my_fp64) atomicAdd(&ctr->tau_fp64, my_fp64);
    }
}

void launch_tau_mixed(const Level &L, const FFView &F, int ntiles, const TauParams &P, int variant,
                      DevCounters *ctr, int32_t *near_ij, double *near_tau, long long near_cap, const EdgeList &E,
                      cudaStream_t s)
{
    if (ntiles <= 0) return;
    const MixedTauBounds Q = mixed_tau_params(P);
    static_assert(TAU_VAR_T[0] == 64 && TAU_VAR_T[1] == 128 && TAU_VAR_T[2] == 64 && TAU_VAR_S[2] == 2 &&
                      TAU_VAR_T[3] == 256,
                  "tau variants");
    if (variant == 0)
        launch_next(k_tau_mixed<64, 1, 1, false>, ntiles, 64, 0, s, L, F, P, Q, ctr, near_ij, near_tau, near_cap, E);
    else if (variant == 1)
        launch_next(k_tau_mixed<128, 1, 1, false>, ntiles, 128, 0, s, L, F, P, Q, ctr, near_ij, near_tau, near_cap, E);
    else if (variant == 2)
        launch_next(k_tau_mixed<64, 2, 1, false>, ntiles, 128, 0, s, L, F, P, Q, ctr, near_ij, near_tau, near_cap, E);
    else
        launch_next(k_tau_mixed<256, 1, 2, false>, ntiles, 128, 0, s, L, F, P, Q, ctr, near_ij, near_tau, near_cap, E);
    CC_COUNT_LAUNCH(1);
}

// the same over a caller's FP64 arrays as one set, hooked into `parent`: 256-wide
// tiles from where they are the faster ones (whole call, 256 / 64-wide: 2048
// bodies 109 / 79 us, 3072 109 / 112, 4096 113 / 129, 8192 136 / 193)
constexpr int TAU_RAW_WIDE_N = 3072;

void launch_tau_raw(const double *m, const double *x3, const double *v3, int n, const TauParams &P, int32_t *parent,
                    DevCounters *ctr, cudaStream_t s)
{
    Level L{};
    double *x = const_cast<double *>(x3), *v = const_cast<double *>(v3);
    const size_t N = (size_t)n;
    L.x = x; L.y = x + N; L.z = x + 2 * N;
    L.vx = v; L.vy = v + N; L.vz = v + 2 * N;
    L.m = const_cast<double *>(m);
    L.parent = parent;
    L.total = n;
    const MixedTauBounds Q = mixed_tau_params(P);
    const FFView F{};
    const EdgeList E{nullptr, nullptr, 0};
    if (n >= TAU_RAW_WIDE_N) {
        const int nt = (n + 255) / 256;
        k_tau_mixed<256, 1, 2, true><<<nt * (nt + 1) / 2, 128, 0, s>>>(L, F, P, Q, ctr, nullptr, nullptr, 0, E);
    } else {
        const int nt = (n + 63) / 64;
        k_tau_mixed<64, 2, 1, true><<<nt * (nt + 1) / 2, 128, 0, s>>>(L, F, P, Q, ctr, nullptr, nullptr, 0, E);
    }
    CC_COUNT_LAUNCH(1);
}

// ------------------------------------------------------------ kick, FP32
// Works in the root-sorted order of the split (members of a component are
// adjacent; rest-set members are their own components).  Grid: (set,
// i-tile, j-chunk).  Thread r of an i-tile accumulates
// sum_j G m_j (x_j - x_i) |x_j - x_i|^-3 over the chunk's j whose label
// differs in FP32 (groups of MK_GROUP terms, each group sum added with
// compensation); a j-tile whose labels and the i-tile's are
// all one component is skipped whole (sorted order: first == last label
// means a uniform tile).  Partials go to scratch in FP64 unless the set has
// a single chunk, in which case v is updated directly.
//
// What bounds it: the FP32 pipe, ~24 cycles a directed pair and warp; two
// columns at a time in packed FP32 (one issue slot for both) take ~17 issue
// slots a pair where one column at a time took ~27.  Each term and the order
// of the sums are as they were, so are the bits.  65536-body fractal, top
// level (4.3e9 directed pairs): 3.77 -> 3.05 ms.
// PACKED = false is the same operations a column at a time, for levels below
// MK_PACKED_MIN pairs.  A column rounds alike in both, but the launch shapes do
// not sum alike (a chunk is a partial sum), the tuner chooses between them by
// their times, and packed arithmetic favours the long chunk by 3 to 8 %: the
// choice turns with it where the two are close, and another choice moves the last
// bits of a kick, which a hard binary magnifies by 1e4 and more before the step is
// over (1.5e-8 of the velocities).  Chunk 4 against 1, time per pair, a column at a
// time / packed: 2^25 pairs 1.055 / 0.988, 2^26 0.990 / 0.988, 2^27 0.958 / 0.947, 2^28
// 0.952 / 0.933, 2^28.9 0.932 / 0.921, from 2^29 on 0.83-0.94 / 0.79-0.93.  What the line
// costs below it: a kick of every pair of 8192 bodies takes 78 us where the packed
// form would take 68, 16384 262 and 213, 32000 946 and 770.
constexpr int MK_T = 128;
constexpr int MK_CHUNK_MAX = 4;  // j-tiles per chunk (tuned per size bin)
static_assert(MK_VAR_CHUNK[0] <= MK_CHUNK_MAX && MK_VAR_CHUNK[1] <= MK_CHUNK_MAX && MK_VAR_CHUNK[2] <= MK_CHUNK_MAX,
              "chunk variants");
constexpr int MK_GROUP = 8;       // j terms summed in plain FP32 per compensated addition

struct __align__(16) MixedKickSmem {
    float4 pq[2][2 * MK_T];  // the kick's copy (k_prep_kick), two stages
    int32_t lab[2][MK_T];
    int32_t cj[MK_T];        // centre-of-mass approximation: the j-tile's eligible components
    int32_t tiles[MK_CHUNK_MAX];
    int32_t apart[MK_CHUNK_MAX];  // 1: no label of the j-tile is one of the i-tile's
    int32_t ntiles;
    uint64_t bar[2];
};

template <bool PACKED>
__device__ __forceinline__ void mk_issue(MixedKickSmem &sm, int st, const FFView &F, const int32_t *label,
                                         int j0, int jn)
{
    const unsigned cnt = (unsigned)((jn + 3) & ~3);
    fence_proxy_async_smem();
    // (packed, an odd last body brings its neighbour's slot along: not added)
    const unsigned bytes = PACKED ? (unsigned)((jn + 1) / 2) * 64u : (unsigned)jn * 32u;
    mbar_expect_tx(&sm.bar[st], bytes + cnt * 4u);
    tma_load_1d(sm.pq[st], F.pq + 2 * (size_t)j0, bytes, &sm.bar[st]);
    tma_load_1d(sm.lab[st], label + j0, cnt * 4u, &sm.bar[st]);
}

// Block = MK_T threads = (MK_T / S rows of the i-tile) x (S column slices of
// each j-tile); the S partial sums of a row are combined in slice order.
// COM: pairs of two far components (ComView, the centre-of-mass
// approximation) are left out, as in the FP64 kick.
template <int S, bool COM, bool PACKED>
__global__ void __launch_bounds__(MK_T) k_kick_mixed(Level L, FFView F, const int32_t *order, const int32_t *koff,
                                                      int chunk, float eps2, double h, DevCounters *ctr,
                                                      double *partial, ComView cv)
{
    pdl_begin();
    constexpr int R = MK_T / S;  // i rows per block
    static_assert(R % 32 == 0, "one slice per warp");
    __shared__ MixedKickSmem sm;
    __shared__ double red[S > 1 ? S : 1][3][R];
    const int tid = threadIdx.x, row = tid % R, slice = tid / R;
    int lo = 0, hi = L.nsets;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (koff[mid] <= (int)blockIdx.x) lo = mid; else hi = mid;
    }
    const int s = lo;
    const int b = blockIdx.x - koff[s];
    const int n = L.set_n[s], start = L.set_start[s];
    const int ntile = (n + MK_T - 1) / MK_T;
    const int nchunk = (ntile + chunk - 1) / chunk;
    const int ti = b / nchunk, ch = b % nchunk;
    const int tj0 = ch * chunk, tj1 = min(ntile, tj0 + chunk);
    const int il = ti * R + row;
    const bool iv = il < n;
    const int t = start + il;  // position in the sorted order
    const int32_t *label = L.klab;
    if (tid == 0) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        fence_mbar_init();
        // tiles with at least one cross-component pair
        const int ia = start + ti * R, ib = start + min(n, (ti + 1) * R) - 1;
        const bool iu = label[ia] == label[ib];
        int q = 0;
        for (int tj = tj0; tj < tj1; ++tj) {
            const int ja = start + tj * MK_T, jb = start + min(n, (tj + 1) * MK_T) - 1;
            if (iu && label[ja] == label[jb] && label[ja] == label[ia]) continue;
            // labels ascend within a set: disjoint ranges share no component
            sm.apart[q] = (label[jb] < label[ia] || label[ib] < label[ja]) ? 1 : 0;
            sm.tiles[q++] = tj;
        }
        sm.ntiles = q;
    }
    __syncthreads();
    const int nt = sm.ntiles;
    if (tid == 0 && nt > 0) mk_issue<PACKED>(sm, 0, F, label, start + sm.tiles[0] * MK_T, min(MK_T, n - sm.tiles[0] * MK_T));
    uint64_t nh[3] = {0, 0, 0}, nl[3] = {0, 0, 0};  // minus the row's position, twice each
    float4 ip0 = make_float4(0, 0, 0, 0), ip1 = ip0;  // the row's position, a column at a time
    int li = 0, ci = -1;
    if (iv) {
        if constexpr (PACKED) {
            const float *q = kick_slot(F, t);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                nh[c] = pack2(-q[2 * c], -q[2 * c]);
                nl[c] = pack2(-q[8 + 2 * c], -q[8 + 2 * c]);
            }
        } else {
            ip0 = F.pq[2 * t];
            ip1 = F.pq[2 * t + 1];
        }
        li = label[t];
        if constexpr (COM) ci = cv.cl[order[t]];
    }
    long long fo = 0;
    int Ks = 0;
    bool iany = false;
    if constexpr (COM) {
        fo = cv.foff[s];
        Ks = cv.K[s];
        iany = __syncthreads_or(ci >= 0) != 0;
    }
    float sx = 0.f, sy = 0.f, sz = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
    bool ok = true;
    for (int q = 0; q < nt; ++q) {
        const int tj = sm.tiles[q], st = q & 1;
        if (tid == 0 && q + 1 < nt) {
            const int tn = sm.tiles[q + 1];
            mk_issue<PACKED>(sm, st ^ 1, F, label, start + tn * MK_T, min(MK_T, n - tn * MK_T));
        }
        const bool got = mbar_wait(&sm.bar[st], (q >> 1) & 1, TMA_WAIT_CYCLES);
        if (__syncthreads_or(!got)) {
            ok = false;
            break;
        }
        const int jn = min(MK_T, n - tj * MK_T);
        bool fchk = false;  // far pairs possible in this tile
        if constexpr (COM) {
            int c = -1;
            if (tid < jn) c = cv.cl[order[start + tj * MK_T + tid]];
            sm.cj[tid] = c;
            fchk = (__syncthreads_or(c >= 0) != 0) && iany;
        }
        if (iv) {
            // g += G m_j r^-3 (x_j - x_i) over groups of MK_GROUP j in plain
            // FP32 (fused), each group sum then added to the compensated
            // total: the per-term roundings dominate the error either way,
            // and the compensation costs 4 operations per component
            float gx, gy, gz;
            // columns k, k + 1 (k even) side by side in packed FP32, added one
            // after the other (two: whether the second exists)
            const ulonglong2 *J = reinterpret_cast<const ulonglong2 *>(sm.pq[st]);
            const uint64_t e2 = pack2(eps2, eps2), mh = pack2(-0.5f, -0.5f), c15 = pack2(1.5f, 1.5f);
            auto pair = [&](int k, bool check, bool two) {
                const ulonglong2 a = J[2 * k], b = J[2 * k + 1], c = J[2 * k + 2];
                const uint64_t lz = J[2 * k + 3].x;
                const uint64_t dx = add2(add2(a.x, nh[0]), add2(c.x, nl[0]));
                const uint64_t dy = add2(add2(a.y, nh[1]), add2(c.y, nl[1]));
                const uint64_t dz = add2(add2(b.x, nh[2]), add2(lz, nl[2]));
                const uint64_t r2 = fma2(dz, dz, fma2(dy, dy, fma2(dx, dx, e2)));
                float ra, rb, wa, wb;
                unpack2(r2, ra, rb);
                uint64_t ri = pack2(rsqrt_ftz(ra), rsqrt_ftz(rb));
                ri = mul2(ri, fma2(mul2(mh, r2), mul2(ri, ri), c15));  // one Newton step
                const uint64_t w = mul2(b.y, mul2(mul2(ri, ri), ri));    // G m_j / r^3
                unpack2(w, wa, wb);
                if (check) {  // same component (and self)
                    if (sm.lab[st][k] == li) wa = 0.f;
                    if (sm.lab[st][k + 1] == li) wb = 0.f;
                }
                if constexpr (COM) {
                    const int c0 = sm.cj[k], c1 = sm.cj[k + 1];
                    if (fchk && ci >= 0 && c0 >= 0 && cv.far[fo + (long long)ci * Ks + c0]) wa = 0.f;
                    if (fchk && ci >= 0 && c1 >= 0 && cv.far[fo + (long long)ci * Ks + c1]) wb = 0.f;
                }
                float xa, xb, ya, yb, za, zb;
                unpack2(dx, xa, xb);
                unpack2(dy, ya, yb);
                unpack2(dz, za, zb);
                gx = fmaf(wa, xa, gx);
                gy = fmaf(wa, ya, gy);
                gz = fmaf(wa, za, gz);
                if (two) {
                    gx = fmaf(wb, xb, gx);
                    gy = fmaf(wb, yb, gy);
                    gz = fmaf(wb, zb, gz);
                }
            };
            // one column
            auto term = [&](int k, bool check) {
                const float4 jp0 = sm.pq[st][2 * k], jp1 = sm.pq[st][2 * k + 1];
                const float dx = (jp0.x - ip0.x) + (jp1.x - ip1.x);
                const float dy = (jp0.y - ip0.y) + (jp1.y - ip1.y);
                const float dz = (jp0.z - ip0.z) + (jp1.z - ip1.z);
                const float r2 = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, eps2)));
                float ri = rsqrtf(r2);
                ri = ri * fmaf(-0.5f * r2, ri * ri, 1.5f);  // one Newton step
                float w = jp0.w * (ri * ri * ri);            // G m_j / r^3
                if (check && sm.lab[st][k] == li) w = 0.f;  // same component (and self)
                if constexpr (COM) {
                    const int c = sm.cj[k];
                    if (fchk && ci >= 0 && c >= 0 && cv.far[fo + (long long)ci * Ks + c]) w = 0.f;
                }
                gx = fmaf(w, dx, gx);
                gy = fmaf(w, dy, gy);
                gz = fmaf(w, dz, gz);
            };
            auto flush = [&]() {
                kahan_add(sx, cx, gx);
                kahan_add(sy, cy, gy);
                kahan_add(sz, cz, gz);
            };
            auto run = [&](bool check) {
                int k = slice * (MK_T / S);
                const int k1 = min(jn, k + MK_T / S);
                for (; k + MK_GROUP <= k1; k += MK_GROUP) {
                    gx = gy = gz = 0.f;
#pragma unroll
                    for (int u = 0; u < MK_GROUP; u += PACKED ? 2 : 1) {
                        if constexpr (PACKED) pair(k + u, check, true);
                        else term(k + u, check);
                    }
                    flush();
                }
                if (k < k1) {
                    gx = gy = gz = 0.f;
                    for (; k < k1; k += PACKED ? 2 : 1) {
                        if constexpr (PACKED) pair(k, check, k + 1 < k1);
                        else term(k, check);
                    }
                    flush();
                }
            };
            if (sm.apart[q]) run(false);
            else run(true);
        }
        __syncthreads();
    }
    if (!ok) {
        raise_err(ctr, DERR_TMA_TIMEOUT);
        mbar_wait(&sm.bar[0], 0, TMA_WAIT_CYCLES);
        mbar_wait(&sm.bar[1], 0, TMA_WAIT_CYCLES);
        return;
    }
    double ax = (double)sx - (double)cx, ay = (double)sy - (double)cy, az = (double)sz - (double)cz;
    if constexpr (S > 1) {
        red[slice][0][row] = ax;
        red[slice][1][row] = ay;
        red[slice][2][row] = az;
        __syncthreads();
        if (slice != 0) return;
        for (int q = 1; q < S; ++q) {
            ax += red[q][0][row];
            ay += red[q][1][row];
            az += red[q][2][row];
        }
    }
    if (!iv) return;
    if (nchunk == 1) {
        const int k = order[t];
        L.vx[k] += h * ax;
        L.vy[k] += h * ay;
        L.vz[k] += h * az;
    } else {
        // partial[(chunk * 3 + c) * cap + t]
        const size_t cap = (size_t)F.cap;
        partial[((size_t)ch * 3 + 0) * cap + t] = ax;
        partial[((size_t)ch * 3 + 1) * cap + t] = ay;
        partial[((size_t)ch * 3 + 2) * cap + t] = az;
    }
}

// Sum the chunk partials of multi-chunk sets (FP64), v += h a.  KR_LANES
// lanes per body: lane s sums chunks s, s + KR_LANES, ... in order, then a
// fixed butterfly combines the lanes, so the rounding order is fixed (run to
// run identical) and the dependent FP64 chain is nchunk/KR_LANES + 3 adds
// long instead of nchunk (an FP64 add's latency dominates this kernel).
constexpr int KR_LANES = 8;

__global__ void k_kick_reduce(Level L, FFView F, const int32_t *order, int chunk, double h, const double *partial,
                              const int32_t *root, double drift_dt)
{
    pdl_begin();
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int t = (int)(g / KR_LANES), sub = (int)(g % KR_LANES);
    int k = -1, nchunk = 1;
    if (t < L.total) {
        k = order[t];
        if (L.sidx[k] >= 0) {
            const int n = L.set_n[L.sidx[k]];
            nchunk = ((n + MK_T - 1) / MK_T + chunk - 1) / chunk;
        }
    }
    const bool on = k >= 0 && L.sidx[k] >= 0 && nchunk > 1;
    const size_t cap = (size_t)F.cap;
    double ax = 0.0, ay = 0.0, az = 0.0;
    if (on) {
        for (int c = sub; c < nchunk; c += KR_LANES) {
            ax += partial[((size_t)c * 3 + 0) * cap + t];
            ay += partial[((size_t)c * 3 + 1) * cap + t];
            az += partial[((size_t)c * 3 + 2) * cap + t];
        }
    }
#pragma unroll
    for (int o = KR_LANES / 2; o > 0; o >>= 1) {
        ax += __shfl_xor_sync(0xffffffffu, ax, o);
        ay += __shfl_xor_sync(0xffffffffu, ay, o);
        az += __shfl_xor_sync(0xffffffffu, az, o);
    }
    if (on && sub == 0) {
        L.vx[k] += h * ax;
        L.vy[k] += h * ay;
        L.vz[k] += h * az;
    }
    // drift_dt > 0: the level's second drift of rest-set members, after their
    // kick (the kick kernels read the float-float copy, never x)
    if (drift_dt > 0.0 && sub == 0 && k >= 0 && L.gid[k] >= 0 && L.cnt[root[k]] == 1) {
        L.x[k] = __dadd_rn(L.x[k], __dmul_rn(drift_dt, L.vx[k]));
        L.y[k] = __dadd_rn(L.y[k], __dmul_rn(drift_dt, L.vy[k]));
        L.z[k] = __dadd_rn(L.z[k], __dmul_rn(drift_dt, L.vz[k]));
    }
}

int mixed_kick_blocks(int n, int chunk, int slices)
{
    const int ntile = (n + MK_T - 1) / MK_T, rows = MK_T / slices;
    return ((n + rows - 1) / rows) * ((ntile + chunk - 1) / chunk);
}

int mixed_kick_chunks(int n, int chunk)
{
    const int ntile = (n + MK_T - 1) / MK_T;
    return (ntile + chunk - 1) / chunk;
}

void launch_kick_mixed(const Level &L, const FFView &F, const int32_t *order, const int32_t *koff, int nblocks,
                       int chunk, int slices, bool multi_chunk, double eps2, double h, DevCounters *ctr,
                       double *partial, const int32_t *root, double drift_dt, bool packed, cudaStream_t s, const ComView *com)
{
    if (nblocks > 0) {
        const ComView cv = com ? *com : ComView{nullptr, nullptr, nullptr, nullptr};
        const float e2 = (float)eps2;
        // (levels of packed size have far more blocks than the sliced shape is for)
        auto k = packed ? (com ? k_kick_mixed<1, true, true> : k_kick_mixed<1, false, true>)
                 : slices == 4 ? (com ? k_kick_mixed<4, true, false> : k_kick_mixed<4, false, false>)
                               : (com ? k_kick_mixed<1, true, false> : k_kick_mixed<1, false, false>);
        launch_next(k, nblocks, MK_T, 0, s, L, F, order, koff, chunk, e2, h, ctr, partial, cv);
        CC_COUNT_LAUNCH(1);
    }
    if ((multi_chunk && nblocks > 0) || (drift_dt > 0.0 && L.total > 0)) {
        const long long threads = (long long)L.total * KR_LANES;
        launch_next(k_kick_reduce, (unsigned)((threads + 255) / 256), 256, 0, s, L, F, order, multi_chunk ? chunk : 1 << 30, h,
                                                                        partial, root, drift_dt);
        CC_COUNT_LAUNCH(1);
    }
}

}  // namespace cc
