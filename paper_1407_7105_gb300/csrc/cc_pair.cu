// cc_pair.cu -- pairwise kernels of the CC split (arXiv:1407.7105):
//   * tau(i,j) in FP64 over all pairs of a set fused with the edge test
//     tau < h (Sec. 2.2), for a time-step graph whose near_tol is wider than
//     the certified kernel's bounds, and the edge list itself;
//   * a first half's edges from its parent's records;
//   * the kick K_{h,V_ij} between members of different components
//     (Eqs. kickij, kickji; Sec. 2.2 K_{h, V_R + V_CC + V_CR}) in FP64: rows
//     in place (k_kick64), or from 2^21 pairs each pair's force once
//     (k_pair_forces) and the rows summed after it (k_kick_rows);
//   * the energy diagnostic H (Eq. Hamiltonian).
// j-tiles are staged in shared memory by TMA bulk copies (cp.async.bulk)
// completing on an mbarrier; every wait is bounded.
#include "cc_device.cuh"
#include "cc_fp64.cuh"
#include <algorithm>

namespace cc {

// ------------------------------------------------------------ helpers
__device__ __forceinline__ int find_set(const int32_t *off, int nsets, int b)
{
    int lo = 0, hi = nsets;  // off[lo] <= b < off[hi]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (off[mid] <= b) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void k_init_parent(int32_t *parent, int32_t *cnt, int total, unsigned long long *edge_count)
{
    pdl_begin();
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < total) {
        parent[k] = k;
        cnt[k] = 0;
    }
    if (k == 0 && edge_count) *edge_count = 0ull;
}

void launch_init_parent(const Level &L, unsigned long long *edge_count, cudaStream_t s)
{
    if (L.total <= 0) return;
    launch_next(k_init_parent, (L.total + 255) / 256, 256, 0, s, L.parent, L.cnt, L.total, edge_count);
    CC_COUNT_LAUNCH(1);
}

// ------------------------------------------------------------ tau + hook
// One CTA per (set, i-tile, j-tile) with i-tile <= j-tile: TAU_T threads,
// thread r owns particle i = i-tile*TAU_T + r and tests it against the
// j-tile staged in shared memory (pairs i < j only).
constexpr int TAU_T = 128;  // tile of the edge-list variant

template <int T>
struct __align__(16) TauSmem {
    double col[7][T + 4];  // x y z vx vy vz m of the j-tile
    uint64_t bar;
};

__device__ __forceinline__ void log_pair(const TauParams &P, double tau, int gi, int gj, DevCounters *ctr,
                                         int32_t *near_ij, double *near_tau, long long near_cap)
{
    if (fabs(tau - P.h) < P.near_tol * P.h) {
        unsigned long long k = atomicAdd(&ctr->near_pairs, 1ull);
        if ((long long)k < near_cap) {
            near_ij[2 * k] = gi < gj ? gi : gj;
            near_ij[2 * k + 1] = gi < gj ? gj : gi;
            near_tau[k] = tau;
        }
    }
}

template <int T>
__global__ void __launch_bounds__(T) k_tau_hook(Level L, TauParams P, DevCounters *ctr, int32_t *near_ij,
                                                     double *near_tau, long long near_cap)
{
    __shared__ TauSmem<T> sm;
    const int tid = threadIdx.x;
    const int s = find_set(L.tile_off, L.nsets, blockIdx.x);
    int t = blockIdx.x - L.tile_off[s];
    const int n = L.set_n[s], start = L.set_start[s];
    const int nt = (n + T - 1) / T;
    int ti = 0;
    while (t >= nt - ti) {
        t -= nt - ti;
        ++ti;
    }
    const int tj = ti + t;
    const int j0 = start + tj * T;
    const int jn = min(T, n - tj * T);

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
        const unsigned bytes = (unsigned)((jn + 3) & ~3) * 8u;
        mbar_expect_tx(&sm.bar, 7u * bytes);
        const double *src[7] = {L.x, L.y, L.z, L.vx, L.vy, L.vz, L.m};
        if (!no_copy) {
#pragma unroll
            for (int c = 0; c < 7; ++c) tma_load_1d(sm.col[c], src[c] + j0, bytes, &sm.bar);
        }
    }
    const int il = ti * T + tid;
    const bool iv = il < n;
    const int i = start + il;
    double xi = 0, yi = 0, zi = 0, vxi = 0, vyi = 0, vzi = 0, mi = 0;
    int gi = -1;
    if (iv) {
        xi = L.x[i]; yi = L.y[i]; zi = L.z[i];
        vxi = L.vx[i]; vyi = L.vy[i]; vzi = L.vz[i];
        mi = L.m[i];
        gi = L.gid[i];
    }
    if (!mbar_wait(&sm.bar, 0, wait_cycles)) {
        raise_err(ctr, DERR_TMA_TIMEOUT);
        // let a copy still in flight land before the CTA exits
        mbar_wait(&sm.bar, 0, wait_cycles);
        return;
    }
    // fault_test = 2: every hook gives up at once (a test of the retry cap)
    const int uf_retry = P.fault_test == 2 ? 0 : UF_RETRY_MAX;
    unsigned long long my_edges = 0;
    if (iv) {
        const int kbeg = (ti == tj) ? tid + 1 : 0;
        auto tau_of = [&](int k) {
            return tau_fp64(__dsub_rn(xi, sm.col[0][k]), __dsub_rn(yi, sm.col[1][k]), __dsub_rn(zi, sm.col[2][k]),
                            __dsub_rn(vxi, sm.col[3][k]), __dsub_rn(vyi, sm.col[4][k]), __dsub_rn(vzi, sm.col[5][k]),
                            mi, sm.col[6][k], P);
        };
        // two pairs' tau in flight (its square roots and divisions are long
        // dependent chains); the second of the last pair may be a repeat
        double tnext = 0.0;
        for (int k = kbeg; k < jn; ++k) {
            double tau;
            if (((k - kbeg) & 1) == 0) {
                tau = tau_of(k);
                tnext = tau_of(k + 1 < jn ? k + 1 : k);
            } else {
                tau = tnext;
            }
            const int j = j0 + k;
            log_pair(P, tau, gi, L.gid[j], ctr, near_ij, near_tau, near_cap);
            if (tau < P.h) {
                ++my_edges;
                if (!uf_union(L.parent, i, j, uf_retry)) raise_err(ctr, DERR_UF_RETRY);
            }
        }
    }
    // warp-aggregated edge count: one atomic per warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) my_edges += __shfl_down_sync(0xffffffffu, my_edges, o);
    if ((tid & 31) == 0 && my_edges) atomicAdd(&ctr->edges, my_edges);
}

// ------------------------------------------------------------ first-half split
// The split of a component's first half (pivot h) sees the state its
// parent split saw at 2h, so tau(i,j) is unchanged: the edges are the
// parent's records that are edges at h, and every pair near h is a parent
// record too (tau < 2h).  Two passes:
//   k_edges_filter, one thread per parent record: records of components the
//   gather did not move to this level (small, Kepler) are skipped (inv[a] is
//   only meaningful where this level's src points back to a); the record's
//   edge depth comes from its e, else its FP64 tau, else (an FP32-certified
//   edge of a fresh mixed split) from certified FP32 decisions at 2h, h,
//   h/2, ... on the parent's float-float copy, which the first half leaves
//   untouched, continued from the parent level's FP64 state at the first
//   undecided threshold (tau_wide, then the FP64 tau); near-threshold pairs
//   are logged, and the edges at h become this split's records (depth carried
//   on, so deeper first halves never need a float-float copy);
//   k_edges_hook: union-find hooking of this split's records, a compact list
//   (a fraction of the parent's), so the pointer chasing of the hooks runs
//   in about one wave (the list holds at least as many records as the
//   parent's, so none is dropped).  The filter pass also points each edge's larger
//   endpoint at its smallest neighbour (atomicMin): every union-find
//   invariant holds for that forest, and in a dense core, where many edges
//   share an endpoint, it spares the hooks their compare-and-swap retries.
__global__ void k_edges_filter(EdgeList PE, long long pcount, Level PL, FFView PF, MixedTauParams Q, int mixed,
                               const int32_t *inv, Level C, EdgeList CE, TauParams P, DevCounters *ctr,
                               int32_t *near_ij, double *near_tau, long long near_cap)
{
    pdl_begin();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long my_edges = 0, my_evals = 0;
    if (t < pcount) {
        const EdgeRec r = PE.rec[t];
        const int a = inv[r.a], b = inv[r.b];
        const bool in = a >= 0 && a < C.total && b >= 0 && b < C.total && C.src[a] == r.a && C.src[b] == r.b &&
                        C.gid[a] >= 0 && C.gid[b] >= 0;
        if (in) {
            const double hp = 2.0 * P.h;  // the parent's pivot
            double tau = r.tau;
            int e = r.e;
            if (e < 0 && tau == tau) e = first_level_at_or_below(tau, hp, EDGE_E_INF);
            if (e < 0) {
                int m = 1, dec = 1;
                if (mixed) {
                    // the tau kernel's decision at hp, restated at hp 2^-m
                    const float4 ip0 = PF.pq[2 * r.a], ip1 = PF.pq[2 * r.a + 1];
                    const float4 iv0 = PF.vq[2 * r.a], iv1 = PF.vq[2 * r.a + 1];
                    const float4 jp0 = PF.pq[2 * r.b], jp1 = PF.pq[2 * r.b + 1];
                    const float4 jv0 = PF.vq[2 * r.b], jv1 = PF.vq[2 * r.b + 1];
                    const float cX = 11.f * U32 * U32 * PF.maxes[0];
                    const float cV = 11.f * U32 * U32 * PF.maxes[1];
                    const TauPrep32 tp = tau_prep_fp32(
                        (jp0.x - ip0.x) + (jp1.x - ip1.x), (jp0.y - ip0.y) + (jp1.y - ip1.y),
                        (jp0.z - ip0.z) + (jp1.z - ip1.z), (jv0.x - iv0.x) + (jv1.x - iv1.x),
                        (jv0.y - iv0.y) + (jv1.y - iv1.y), (jv0.z - iv0.z) + (jv1.z - iv1.z), ip0.w + jp0.w, cX, cV,
                        Q);
                    while (m < 100) {
                        dec = tau_decide_at(tp, Q.etah * pow2f(m));
                        if (dec != 1) break;
                        ++m;
                    }
                }
                if (mixed && dec == 0) {
                    e = m;
                } else {
                    const int i = r.a, j = r.b;
                    const TauOpen o = tau_open(__dsub_rn(PL.x[i], PL.x[j]), __dsub_rn(PL.y[i], PL.y[j]),
                                               __dsub_rn(PL.z[i], PL.z[j]), __dsub_rn(PL.vx[i], PL.vx[j]),
                                               __dsub_rn(PL.vy[i], PL.vy[j]), __dsub_rn(PL.vz[i], PL.vz[j]),
                                               PL.m[i], PL.m[j], P, hp, m, EDGE_E_INF);
                    if (o.e >= 0) {
                        e = o.e;
                    } else {
                        tau = o.tau;
                        ++my_evals;
                        const int e64 = first_level_at_or_below(tau, hp, EDGE_E_INF);
                        e = e64 > m ? e64 : m;
                    }
                }
            }
            if (tau == tau) log_pair(P, tau, C.gid[a], C.gid[b], ctr, near_ij, near_tau, near_cap);
            if (e >= 2) {
                ++my_edges;
                // link the larger endpoint to its smallest neighbour so far:
                // a forest with parent < self whose links are edges, built
                // without retries; the hook pass then finds most record
                // endpoints already in one tree
                atomicMin(&C.parent[max(a, b)], min(a, b));
                // the host sizes this list to the parent's record count, so
                // a record is never dropped (the hook pass must see every edge)
                if (!record_edge(CE, min(a, b), max(a, b), e >= EDGE_E_INF ? EDGE_E_INF : e - 1, tau))
                    raise_err(ctr, DERR_UF_RETRY);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_edges += __shfl_down_sync(0xffffffffu, my_edges, o);
        my_evals += __shfl_down_sync(0xffffffffu, my_evals, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (my_edges) atomicAdd(&ctr->edges, my_edges);
        if (my_evals) {
            atomicAdd(&ctr->tau_fp64, my_evals);
            atomicAdd(&ctr->tau_evals, my_evals);
        }
    }
}

__global__ void k_edges_hook(EdgeList E, int32_t *parent, DevCounters *ctr)
{
    pdl_begin();
    const long long n = (long long)min(*E.count, (unsigned long long)E.cap);
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const EdgeRec r = E.rec[t];
        // a shared parent, or the link itself, already puts a and b in one
        // tree (a parent is an ancestor, and trees only merge)
        const int pa = __ldca(parent + r.a), pb = __ldca(parent + r.b);
        if (pa == pb || pb == r.a || pa == r.b) continue;
        if (!uf_union_ca(parent, r.a, r.b)) raise_err(ctr, DERR_UF_RETRY);
    }
}

void launch_edges_reuse(const EdgeList &parent, long long pcount, const Level &PL, const FFView &PF, bool mixed,
                        const int32_t *inv, const Level &C, const EdgeList &child, const TauParams &P,
                        DevCounters *ctr, int32_t *near_ij, double *near_tau, long long near_cap, cudaStream_t s,
                        bool hook)
{
    if (pcount <= 0) return;
    const double hp = 2.0 * P.h;
    TauParams PP = P;
    PP.h = hp;
    const MixedTauParams Q = mixed_tau_params(PP);
    const unsigned blocks = (unsigned)((pcount + 255) / 256);
    launch_next(k_edges_filter, blocks, 256, 0, s, parent, pcount, PL, PF, Q, mixed ? 1 : 0, inv, C, child, P, ctr, near_ij,
                                          near_tau, near_cap);
    CC_COUNT_LAUNCH(1);
    if (hook) {
        // the hooks: at most pcount records, usually far fewer (grid-stride)
        launch_next(k_edges_hook, blocks < 1216u ? blocks : 1216u, 256, 0, s, child, C.parent, ctr);
        CC_COUNT_LAUNCH(1);
    }
}

// Edge-list variant for the time-step-graph entry point: same predicate,
// each edge written as (gid_i, gid_j), gid_i < gid_j, at an atomically
// reserved slot (order fixed afterwards by a sort).
__global__ void __launch_bounds__(TAU_T) k_tau_edges(Level L, TauParams P, DevCounters *ctr, int32_t *edges,
                                                      long long edge_cap, int32_t *near_ij, double *near_tau,
                                                      long long near_cap)
{
    __shared__ TauSmem<TAU_T> sm;
    const int tid = threadIdx.x;
    const int s = find_set(L.tile_off, L.nsets, blockIdx.x);
    int t = blockIdx.x - L.tile_off[s];
    const int n = L.set_n[s], start = L.set_start[s];
    const int nt = (n + TAU_T - 1) / TAU_T;
    int ti = 0;
    while (t >= nt - ti) {
        t -= nt - ti;
        ++ti;
    }
    const int tj = ti + t;
    const int j0 = start + tj * TAU_T;
    const int jn = min(TAU_T, n - tj * TAU_T);
    if (tid == 0) {
        mbar_init(&sm.bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0) {
        const unsigned bytes = (unsigned)((jn + 3) & ~3) * 8u;
        mbar_expect_tx(&sm.bar, 7u * bytes);
        const double *src[7] = {L.x, L.y, L.z, L.vx, L.vy, L.vz, L.m};
#pragma unroll
        for (int c = 0; c < 7; ++c) tma_load_1d(sm.col[c], src[c] + j0, bytes, &sm.bar);
    }
    const int il = ti * TAU_T + tid;
    const bool iv = il < n;
    const int i = start + il;
    double xi = 0, yi = 0, zi = 0, vxi = 0, vyi = 0, vzi = 0, mi = 0;
    int gi = -1;
    if (iv) {
        xi = L.x[i]; yi = L.y[i]; zi = L.z[i];
        vxi = L.vx[i]; vyi = L.vy[i]; vzi = L.vz[i];
        mi = L.m[i];
        gi = L.gid[i];
    }
    if (!mbar_wait(&sm.bar, 0, TMA_WAIT_CYCLES)) {
        raise_err(ctr, DERR_TMA_TIMEOUT);
        mbar_wait(&sm.bar, 0, TMA_WAIT_CYCLES);
        return;
    }
    if (!iv) return;
    const int kbeg = (ti == tj) ? tid + 1 : 0;
    for (int k = kbeg; k < jn; ++k) {
        const double tau = tau_fp64(__dsub_rn(xi, sm.col[0][k]), __dsub_rn(yi, sm.col[1][k]),
                                    __dsub_rn(zi, sm.col[2][k]), __dsub_rn(vxi, sm.col[3][k]),
                                    __dsub_rn(vyi, sm.col[4][k]), __dsub_rn(vzi, sm.col[5][k]), mi,
                                    sm.col[6][k], P);
        const int j = j0 + k;
        const int gj = L.gid[j];
        log_pair(P, tau, gi, gj, ctr, near_ij, near_tau, near_cap);
        if (tau < P.h) {
            if (!uf_union(L.parent, i, j)) raise_err(ctr, DERR_UF_RETRY);
            unsigned long long e = atomicAdd(&ctr->edges, 1ull);
            if ((long long)e < edge_cap) {
                edges[2 * e] = gi < gj ? gi : gj;
                edges[2 * e + 1] = gi < gj ? gj : gi;
            }
        }
    }
}

void launch_tau_hook(const Level &L, int ntiles, const TauParams &P, DevCounters *ctr,
                     int32_t *edges, long long edge_cap, int32_t *near_ij, double *near_tau, long long near_cap,
                     cudaStream_t s)
{
    if (ntiles <= 0) return;
    if (edges) {
        k_tau_edges<<<ntiles, TAU_T, 0, s>>>(L, P, ctr, edges, edge_cap, near_ij, near_tau, near_cap);
        CC_COUNT_LAUNCH(1);
        return;
    }
    k_tau_hook<TAU_T><<<ntiles, TAU_T, 0, s>>>(L, P, ctr, near_ij, near_tau, near_cap);
    CC_COUNT_LAUNCH(1);
}

// ------------------------------------------------------------ kick (FP64)
// One block per KB_R rows of a set's 32-row tile.  For each 32 columns eight
// warps, one a row, compute the row's pair forces into shared memory (a
// skipped pair is an exact +0), while a ninth adds the previous 32 columns',
// one lane a row and component, in ascending j: a_i is the sum over j in
// ascending id, term by term as in the plain definition, so the result is the
// oracle's bit for bit; then v_i += h a_i.
//
// What bounds it: for the small sets that come here the chain of n additions
// (64 cycles each; the forces of 32 columns are ready sooner); a set of 32-row
// blocks left all but n/32 SMs idle, and those FP64-bound.  256 bodies: 78 us
// with 32 rows a block, 18 us now.
constexpr int KB_T = 32;  // the i-tile prefix, and the columns of a step
constexpr int KB_R = 8;   // rows of a block
constexpr int KB_THREADS = 32 * (KB_R + 1);
static_assert(K64_VAR_T[0] == KB_T, "the FP64 kick runs on the 32-body i-tile prefix");

// MODE 1 (centre-of-mass approximation): pairs of far components (ComView)
// are left out; their kick is the centre-of-mass one that launch_com_apply
// adds afterwards.  MODE 2 (OK split): the fast pairs (OkView: each row's
// partners, sorted) are left out, every other pair of the set kicks.
template <int MODE>
__global__ void __launch_bounds__(KB_THREADS) k_kick64(Level L, const int32_t *label, double G, double eps2, double h,
                                                       double one, ComView cv, OkView okv)
{
    pdl_begin();
    __shared__ double f[2][3][KB_R][KB_T + 1];
    const int tile = blockIdx.x / (KB_T / KB_R);
    const int s = find_set(L.itile_off, L.nsets, tile);
    const int n = L.set_n[s], start = L.set_start[s];
    const int il0 = (tile - L.itile_off[s]) * KB_T + (blockIdx.x % (KB_T / KB_R)) * KB_R;
    if (il0 >= n) return;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nk = (n + KB_T - 1) / KB_T;
    if (w == KB_R) {
        // the adding warp: lane = 8 c + r
        const int c = min(lane / KB_R, 2), r = lane % KB_R;
        double acc = 0.0;
        __syncthreads();
        for (int k = 0; k < nk; ++k) {
            const double *t = f[k & 1][c][r];
#pragma unroll
            for (int jj = 0; jj < KB_T; ++jj) acc = add_fma(t[jj], acc, one);
            __syncthreads();
        }
        if (lane < 3 * KB_R && il0 + r < n) {
            const int i = start + il0 + r;
            double *v = c == 0 ? L.vx : (c == 1 ? L.vy : L.vz);
            v[i] = __dadd_rn(v[i], __dmul_rn(h, acc));
        }
        return;
    }
    const bool on = il0 + w < n, soft = eps2 != 0.0;
    const int i = start + (on ? il0 + w : il0);
    const double xi = L.x[i], yi = L.y[i], zi = L.z[i];
    const int li = label[i];
    long long fo = 0;
    int Ks = 0, ci = -1, oq = 0, oe = 0;
    if (MODE == 1) {
        fo = cv.foff[s];
        Ks = cv.K[s];
        ci = cv.cl[i];
    }
    if (MODE == 2) {
        oq = okv.row_ptr[i];
        oe = okv.row_ptr[i + 1];
    }
    for (int k = 0; k < nk; ++k) {
        const int jl = k * KB_T + lane, j = start + min(jl, n - 1);
        bool use = on && jl < n && j != i && label[j] != li;
        if (MODE == 1 && use && ci >= 0) {
            const int c = cv.cl[j];
            if (c >= 0) use = cv.far[fo + (long long)ci * Ks + c] == 0;
        }
        if (MODE == 2) {
            // the row's fast partners among these columns, 32 of its sorted list at a time
            const int jb = start + k * KB_T;
            uint32_t mk = 0u;
            for (;;) {
                const int p = oq + lane < oe ? okv.col[2 * (long long)(oq + lane) + 1] : 0x7fffffff;
                const bool in = p < jb + KB_T;
                mk |= __reduce_or_sync(0xffffffffu, in && p >= jb ? 1u << (p - jb) : 0u);
                const int cnt = __popc(__ballot_sync(0xffffffffu, in));
                oq += cnt;
                if (cnt < 32) break;
            }
            use = use && ((mk >> lane) & 1u) == 0u;
        }
        double t0 = 0.0, t1 = 0.0, t2 = 0.0;
        if (use) {
            const double dx0 = add_fma(L.x[j], -xi, one), dx1 = add_fma(L.y[j], -yi, one),
                         dx2 = add_fma(L.z[j], -zi, one);
            const double gm = __dmul_rn(G, L.m[j]);
            double v;
            const bool fast = pair_rinv3(dx0, dx1, dx2, eps2, soft, one, v) && exp_fast(d2u(gm));
            if (fast) {
                const uint64_t wv = mul_rn(d2u(gm), d2u(v));
                t0 = u2d(mul_rn(wv, d2u(dx0)));
                t1 = u2d(mul_rn(wv, d2u(dx1)));
                t2 = u2d(mul_rn(wv, d2u(dx2)));
            } else {
                const double wv = __dmul_rn(gm, v);
                t0 = __dmul_rn(wv, dx0);
                t1 = __dmul_rn(wv, dx1);
                t2 = __dmul_rn(wv, dx2);
            }
        }
        f[k & 1][0][w][lane] = t0;
        f[k & 1][1][w][lane] = t1;
        f[k & 1][2][w][lane] = t2;
        __syncthreads();
    }
    __syncthreads();  // (the adding warp's last step)
}

// Three n x n matrices per set (components x, y, z) at pf.moff[s]: row j,
// column i = the force G m_j r_ij^-3 (x_j - x_i) of j on i (the diagonal
// unused), so that k_kick_rows, a lane per i, reads them straight.  One block
// per 128-wide triangular tile (TI <= TJ; the grid and prefix L.tile_off of
// the 128-wide tau tiles), in 32 x 32 sub-tiles: every unordered pair is
// evaluated once with the kick's own operations (dx = x_j - x_i; the squares
// make r^2, and so r^-3, the same bits for (j, i), and x_i - x_j = -dx
// exactly); the force on j goes out directly, the force on i through shared
// memory.
//
// What bounds it: the FP64 pipe, one warp instruction in 64 cycles.  Of a
// pair's 18 IEEE operations (more with unequal masses or softening), two of
// them a square root and a reciprocal, the five additions, two residuals and
// two products stay there; the other products and r^-3 run on the integer and
// FP32 pipes meanwhile (cc_fp64.cuh: 66 cycles a product, 300 r^-3).  Equal masses (a sub-tile's warp sees only one): the force on j is
// the negated force on i, bit for bit.  16384 bodies (1.34e8 pairs): 8.6 ms
// with every operation on the FP64 pipe, 2.4 ms so (two of the products left
// on it; none 2.66, one 2.46, three 2.55, four 2.81 ms).
constexpr int KR_T = 32, KR_W = 128, PF_THREADS = 256;
constexpr int PF_Q = KR_T * KR_T / PF_THREADS;  // pairs of a sub-tile per thread
static_assert(KR_T == KB_T, "the force sub-tiles are the kick's i-tiles");
static_assert(KR_W == TAU_VAR_T[TAU_VAR_128], "the force tiles are the 128-wide tau tiles");
template <bool SOFT>
__global__ void __launch_bounds__(PF_THREADS, 6) k_pair_forces(Level L, double G, double eps2, double one, double nzero,
                                                            PairFactors pf)
{
    __shared__ double xi[4][KR_W];  // x, y, z, G m
    __shared__ double xj[4][KR_W];
    __shared__ double t[3][KR_T][KR_T + 1];
    const int tid = threadIdx.x;
    const int s = find_set(L.tile_off, L.nsets, blockIdx.x);
    int tt = blockIdx.x - L.tile_off[s];
    const int n = L.set_n[s], start = L.set_start[s];
    const long long nn = (long long)n * n;
    const int nT = (n + KR_W - 1) / KR_W;
    const int TI = tri_tile_row(tt, nT), TJ = TI + tt;
    const int i0 = TI * KR_W, j0 = TJ * KR_W;
    const int ni = min(KR_W, n - i0), nj = min(KR_W, n - j0);
    double *S = pf.S + pf.moff[s];
    bool in = true;  // every G m in the range of the integer products
    for (int e = tid; e < KR_W; e += PF_THREADS) {
        const bool vi = e < ni, vj = e < nj;
        xi[0][e] = vi ? L.x[start + i0 + e] : 0.0;
        xi[1][e] = vi ? L.y[start + i0 + e] : 0.0;
        xi[2][e] = vi ? L.z[start + i0 + e] : 0.0;
        xi[3][e] = vi ? __dmul_rn(G, L.m[start + i0 + e]) : 1.0;
        xj[0][e] = vj ? L.x[start + j0 + e] : 0.0;
        xj[1][e] = vj ? L.y[start + j0 + e] : 0.0;
        xj[2][e] = vj ? L.z[start + j0 + e] : 0.0;
        xj[3][e] = vj ? __dmul_rn(G, L.m[start + j0 + e]) : 1.0;
        in = in && exp_fast(d2u(xi[3][e])) && exp_fast(d2u(xj[3][e]));
    }
    in = __syncthreads_and(in) != 0;
    for (int a = 0; a < KR_W / KR_T; ++a) {
        for (int b = TI == TJ ? a : 0; b < KR_W / KR_T; ++b) {
            const int il = a * KR_T, jl = b * KR_T;
            if (il >= ni || jl >= nj) continue;  // (uniform over the block)
            __syncthreads();  // (the previous sub-tile's transposed write)
#pragma unroll 1
            for (int q = 0; q < PF_Q; ++q) {
                const int pidx = tid + q * PF_THREADS, ii = pidx >> 5, jj = pidx & 31;
                const int gi = il + ii, gj = jl + jj;
                const bool on = gi < ni && gj < nj && j0 + gj > i0 + gi;
                const uint64_t gmj = d2u(xj[3][gj]), gmi = d2u(xi[3][gi]);
                const bool same = __all_sync(0xffffffffu, !on || gmj == gmi);
                if (!on) continue;
                const double dx0 = add_fma(xj[0][gj], -xi[0][gi], one);
                const double dx1 = add_fma(xj[1][gj], -xi[1][gi], one);
                const double dx2 = add_fma(xj[2][gj], -xi[2][gi], one);
                const uint64_t d2 = d2u(dx2);
                uint64_t w, f0, f1, f2, g0, g1, g2;
                double vd;
                const bool fast = pair_rinv3(dx0, dx1, dx2, eps2, SOFT, one, vd) && in;
                const uint64_t v = d2u(vd);
                if (fast) {
                    // (two of the three products of a force on the FP64 pipe: the
                    // two pipes then finish about together)
                    w = mul_rn(gmj, v);
                    f0 = d2u(__fma_rn(u2d(w), dx0, nzero));
                    f1 = d2u(__fma_rn(u2d(w), dx1, nzero));
                    f2 = mul_rn(w, d2);
                    if (same) {
                        g0 = f0;
                        g1 = f1;
                        g2 = f2;
                    } else {
                        w = mul_rn(gmi, v);
                        g0 = mul_rn(w, d2u(dx0));
                        g1 = mul_rn(w, d2u(dx1));
                        g2 = mul_rn(w, d2);
                    }
                } else {
                    const double wij = __dmul_rn(u2d(gmj), vd), wji = __dmul_rn(u2d(gmi), vd);
                    f0 = d2u(__dmul_rn(wij, dx0));
                    f1 = d2u(__dmul_rn(wij, dx1));
                    f2 = d2u(__dmul_rn(wij, dx2));
                    g0 = d2u(__dmul_rn(wji, dx0));
                    g1 = d2u(__dmul_rn(wji, dx1));
                    g2 = d2u(__dmul_rn(wji, dx2));
                }
                const uint64_t minus = 1ull << 63;
                const long long e = (long long)(i0 + gi) * n + (j0 + gj);
                S[e] = u2d(g0 ^ minus);
                S[nn + e] = u2d(g1 ^ minus);
                S[2 * nn + e] = u2d(g2 ^ minus);
                t[0][ii][jj] = u2d(f0);
                t[1][ii][jj] = u2d(f1);
                t[2][ii][jj] = u2d(f2);
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < PF_Q; ++q) {
                const int pidx = tid + q * PF_THREADS, jj = pidx >> 5, ii = pidx & 31;
                const int gi = il + ii, gj = jl + jj;
                if (gi < ni && gj < nj && j0 + gj > i0 + gi) {
                    const long long e = (long long)(j0 + gj) * n + (i0 + gi);
                    S[e] = t[0][ii][jj];
                    S[nn + e] = t[1][ii][jj];
                    S[2 * nn + e] = t[2][ii][jj];
                }
            }
        }
    }
}

// v_i += h sum_j (force of j on i) from k_pair_forces' matrices, over the j of
// the set in ascending order whose label differs (and, OKM, that are not
// among i's fast partners, which are sorted): the terms and the order of
// k_kick64 (a left-out term is an exact +0), so its bits.
//
// What bounds it: the chain of n additions of a row, one in 64 cycles however
// few rows there are, times the warps on a scheduler (3 for 16384 rows).  A
// warp issues in order, so whatever else it does between two additions comes
// on top (158 cycles a column when one warp also copied and masked its
// columns).  Hence two warps: one takes 32 rows of one component, lane = row,
// and only reads shared memory and adds; its helper copies the columns
// (coalesced 256-byte pieces, 48 columns ahead) and overwrites the left-out
// terms with zero; they meet once per KW columns at a barrier of their own.
// Four pairs a block, so every scheduler gets the same number.  24 bytes a
// pair, 4.7 TB/s at the additions' rate.  The 15 launches of a 16384-body
// step: 8.5 ms when the tiles were staged by 256 threads for 96 to add, 7.7 ms so
// (ncu; the step 19.1 ms).
constexpr int KW = 16;                      // columns a stage
constexpr int KR_PAIRS = 4, KR_STAGES = 4;  // 16 KB a pair
constexpr int KR_SMEM = KR_PAIRS * KR_STAGES * KW * 32 * 8;

// 8 bytes global -> shared, asynchronous (rows of odd n are 8-byte aligned only)
__device__ __forceinline__ void cp_async8(unsigned dst, const double *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

template <bool OKM>
__global__ void __launch_bounds__(64 * KR_PAIRS) k_kick_rows(Level L, const int32_t *label, double h, double one,
                                                             int nitiles, OkView okv, PairFactors pf)
{
    extern __shared__ __align__(16) double ring[];  // [pair][stage][column][lane]
    const int p = (threadIdx.x >> 5) % KR_PAIRS, lane = threadIdx.x & 31;
    const bool adds = threadIdx.x < 32 * KR_PAIRS;
    const int w = blockIdx.x * KR_PAIRS + p, tile = w / 3, c = w % 3;
    if (tile >= nitiles) return;  // (both warps of the pair)
    const int s = find_set(L.itile_off, L.nsets, tile);
    const int n = L.set_n[s], start = L.set_start[s];
    const int il = (tile - L.itile_off[s]) * KB_T + lane;
    const bool on = il < n;
    const int i = start + (on ? il : n - 1);
    double *mine = ring + p * (KR_STAGES * KW * 32) + lane;
    const int nk = (n + KW - 1) / KW;
    // (immediate numbers: a register operand would claim all 16 barriers)
    auto meet = [&]() {
        if (p == 0) asm volatile("bar.sync 1, 64;" ::: "memory");
        else if (p == 1) asm volatile("bar.sync 2, 64;" ::: "memory");
        else if (p == 2) asm volatile("bar.sync 3, 64;" ::: "memory");
        else asm volatile("bar.sync 4, 64;" ::: "memory");
    };
    static_assert(KR_PAIRS == 4, "one barrier a pair");
    if (adds) {
        double acc = 0.0;
        for (int k = 0; k < nk; ++k) {
            meet();  // stage k is ready
            const double *f = mine + (k % KR_STAGES) * (KW * 32);
#pragma unroll
            for (int u = 0; u < KW; ++u) acc = add_fma(f[u * 32], acc, one);
        }
        if (on) {
            double *v = c == 0 ? L.vx : (c == 1 ? L.vy : L.vz);
            v[i] = __dadd_rn(v[i], __dmul_rn(h, acc));
        }
        return;
    }
    const double *F = pf.S + pf.moff[s] + (long long)c * n * n + (i - start);
    const int32_t *lab = label + start;  // (sets start at multiples of four elements)
    const int li = label[i];
    // OKM: the columns of the row's next two fast partners (the second is read
    // long before it is needed)
    int fast = 0x7fffffff, ahead = 0x7fffffff, fq = 0, fe = 0;
    auto next_fast = [&]() {
        fast = ahead;
        ahead = fq < fe ? okv.col[2 * (long long)fq + 1] - start : 0x7fffffff;
        ++fq;
    };
    if (OKM) {
        fq = okv.row_ptr[i];
        fe = okv.row_ptr[i + 1];
        next_fast();
        next_fast();
    }
    const unsigned mine_s = smem_u32(mine);
    auto issue = [&](int k) {
        const unsigned d = mine_s + (k % KR_STAGES) * (KW * 32 * 8);
#pragma unroll
        for (int u = 0; u < KW; ++u) {
            if (k * KW + u < n) cp_async8(d + u * 256, F);
            F += n;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int k = 0; k < KR_STAGES - 1; ++k) issue(k);
    for (int k = 0; k < nk; ++k) {
        const int j = k * KW;
        uint32_t out = 0u;  // the stage's left-out columns
        if (OKM) {
            while (fast < j + KW) {
                out |= 1u << (fast - j);
                next_fast();
            }
        }
        // (past a set's end the labels are its padding's or the next set's, in
        // the same buffer: those columns are left out whatever they hold)
#pragma unroll
        for (int u = 0; u < KW; u += 4) {
            const int4 l = *reinterpret_cast<const int4 *>(lab + j + u);
            out |= (l.x == li ? 1u << u : 0u) | (l.y == li ? 2u << u : 0u) | (l.z == li ? 4u << u : 0u) |
                   (l.w == li ? 8u << u : 0u);
        }
        if (j + KW > n) out |= 0xffffffffu << (n - j);
        asm volatile("cp.async.wait_group %0;" ::"n"(KR_STAGES - 2) : "memory");
        double *f = mine + (k % KR_STAGES) * (KW * 32);
#pragma unroll
        for (int u = 0; u < KW; ++u)
            if (out >> u & 1u) f[u * 32] = 0.0;
        meet();                    // stage k to the adding warp, which is done with stage k - 1
        issue(k + KR_STAGES - 1);  // into that one's place
    }
}

void launch_kick(const Level &L, const int32_t *label, int nitiles, double G, double eps2, double h,
                 cudaStream_t s, const ComView *com, const OkView *okv,
                 const PairFactors *pf)
{
    if (nitiles <= 0) return;
    const ComView nc{nullptr, nullptr, nullptr, nullptr};
    const OkView no{nullptr, nullptr};
    const unsigned grid = (unsigned)nitiles * (KB_T / KB_R);
    const bool pre = pf && pf->S && !(com && com->cl);
    // (the two launched the ordinary way: with the rows' kernel waiting on the SMs
    // beside the forces' last blocks a 16384-body step took 20.8 ms, not 19.4)
    if (pre) {
        if (eps2 != 0.0) k_pair_forces<true><<<pf->nblocks, PF_THREADS, 0, s>>>(L, G, eps2, 1.0, -0.0, *pf);
        else k_pair_forces<false><<<pf->nblocks, PF_THREADS, 0, s>>>(L, G, eps2, 1.0, -0.0, *pf);
        const int nb = (3 * nitiles + KR_PAIRS - 1) / KR_PAIRS;
        if (okv && okv->row_ptr) {
            cudaFuncSetAttribute(k_kick_rows<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, KR_SMEM);
            k_kick_rows<true><<<nb, 64 * KR_PAIRS, KR_SMEM, s>>>(L, label, h, 1.0, nitiles, *okv, *pf);
        } else {
            cudaFuncSetAttribute(k_kick_rows<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, KR_SMEM);
            k_kick_rows<false><<<nb, 64 * KR_PAIRS, KR_SMEM, s>>>(L, label, h, 1.0, nitiles, no, *pf);
        }
        CC_COUNT_LAUNCH(1);
    } else if (okv && okv->row_ptr) {
        launch_next(k_kick64<2>, grid, KB_THREADS, 0, s, L, label, G, eps2, h, 1.0, nc, *okv);
    } else if (com && com->cl) {
        launch_next(k_kick64<1>, grid, KB_THREADS, 0, s, L, label, G, eps2, h, 1.0, *com, no);
    } else {
        launch_next(k_kick64<0>, grid, KB_THREADS, 0, s, L, label, G, eps2, h, 1.0, nc, no);
    }
    CC_COUNT_LAUNCH(1);
}

// ------------------------------------------------------------ energy
constexpr int EN_T = 128;  // rows of a block's tile, one a thread
constexpr int EN_C = 32;   // its columns

// tiles (128 rows x 32 columns) holding a pair i < j; blocks share them in turn
int energy_blocks(long long n, int nsys, int nsm)
{
    const long long nt = (n + EN_T - 1) / EN_T, nc = (n + EN_C - 1) / EN_C;
    const long long tiles = nsys > 1 ? nt : nt * nc - 2 * nt * (nt - 1);
    return (int)std::min<long long>(tiles, 8ll * nsm);
}

// Kinetic and potential energy, momentum and angular momentum.  With
// independent systems (sys_off, nsys + 1 offsets) the potential sums only
// pairs inside one system: systems never interact, so a pair of two
// systems belongs to no system's Hamiltonian.
//
// What bounds it: the FP64 pipe.  A pair's IEEE square root and quotient (~35
// issue slots of 64 cycles with the rest) became r^-1 by rsqrt_near, 0.51 ulp
// off the FP64 pipe but for one residual; left on it are the differences,
// two of r^2's three products, the residual and the sum m_j/r: seven.  One
// system's triangle is cut into tiles of 128 x 32 that the blocks take in
// turn (rows of very different length left the chip to the last of them).
// 65536 bodies (2.1e9 pairs): 141.8 ms before, 27.9 ms now (31.6 with all three
// products of r^2 on the FP64 pipe).
template <bool ONE, bool SOFT>
__global__ void __launch_bounds__(EN_T, 8) k_energy(const double *x3, const double *v3, const double *m,
                                                  long long n, double G, double eps2, double one,
                                                  const int32_t *sys_off, int nsys, double *partial)
{
    __shared__ double2 sxy[EN_C], szm[EN_C];
    __shared__ double red[8][EN_T / 32];
    __shared__ long long blk_hi;
    const long long nt = (n + EN_T - 1) / EN_T, nc = (n + EN_C - 1) / EN_C;
    double q[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    double xi = 0, yi = 0, zi = 0, mi = 0;
    long long i = 0, hi = 0;
    auto take_row = [&](long long b) {  // this thread's body of row tile b, its system's end
        i = b * EN_T + threadIdx.x;
        hi = i < n ? n : 0;
        if (i < n) {
            xi = x3[i]; yi = x3[n + i]; zi = x3[2 * n + i];
            mi = m[i];
            if (!ONE) {
                int lo = 0, up = nsys;  // sys_off[lo] <= i < sys_off[up]
                while (up - lo > 1) {
                    const int mid = (lo + up) >> 1;
                    if ((long long)sys_off[mid] <= i) lo = mid;
                    else up = mid;
                }
                hi = sys_off[up];
            }
        }
    };
    auto single = [&]() {  // the body's own terms, once a row tile
        if (i >= n) return;
        const double vx = v3[i], vy = v3[n + i], vz = v3[2 * n + i];
        q[0] += 0.5 * mi * (vx * vx + vy * vy + vz * vz);
        q[2] += mi * vx; q[3] += mi * vy; q[4] += mi * vz;
        q[5] += mi * (yi * vz - zi * vy);
        q[6] += mi * (zi * vx - xi * vz);
        q[7] += mi * (xi * vy - yi * vx);
    };
    auto columns = [&](long long c) {  // sum of m_j/r over column tile c
        const long long j0 = c * EN_C;
        __syncthreads();
        if (threadIdx.x < EN_C && j0 + threadIdx.x < n) {
            const long long j = j0 + threadIdx.x;
            sxy[threadIdx.x] = make_double2(x3[j], x3[n + j]);
            szm[threadIdx.x] = make_double2(x3[2 * n + j], m[j]);
        }
        __syncthreads();
        const int k0 = (int)max(0ll, i + 1 - j0), k1 = (int)min((long long)EN_C, hi - j0);
        double acc = 0.0;
#pragma unroll 2
        for (int k = 0; k < EN_C; ++k) {
            const double2 a = sxy[k], b = szm[k];
            const double dx = add_fma(a.x, -xi, one), dy = add_fma(a.y, -yi, one), dz = add_fma(b.x, -zi, one);
            const uint64_t dzb = d2u(dz);
            const bool in = k >= k0 && k < k1;
            double r2;
            bool fast = fast_range(dzb);
            if (fast) {
                r2 = fma(dx, dx, fma(dy, dy, u2d(sqr_rn(dzb))));
                if (SOFT) r2 = add_fma(r2, eps2, one);
                fast = exp_fast(d2u(r2));
            }
            double y;
            if (fast) {
                y = u2d(rsqrt_near(d2u(r2)));
            } else {
                y = in ? 1.0 / sqrt(dx * dx + dy * dy + dz * dz + eps2) : 0.0;
            }
            acc = fma(in ? b.y : 0.0, y, acc);
        }
        q[1] -= G * mi * acc;
    };
    if (ONE) {
        long long b = 0, c = blockIdx.x, at = -1;
        for (;; c += gridDim.x) {
            while (b < nt && c >= nc) {
                c += 4 * (b + 1) - nc;
                ++b;
            }
            if (b >= nt) break;
            if (b != at) {
                at = b;
                take_row(b);
            }
            if (c == 4 * b) single();
            columns(c);
        }
    } else {
        for (long long b = blockIdx.x; b < nt; b += gridDim.x) {
            take_row(b);
            single();
            if (threadIdx.x == 0) blk_hi = 0;
            __syncthreads();
            atomicMax((unsigned long long *)&blk_hi, (unsigned long long)hi);
            __syncthreads();
            const long long jend = blk_hi;
            for (long long c = 4 * b; c * EN_C < jend; ++c) columns(c);
            __syncthreads();
        }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        double val = q[c];
        for (int o = 16; o > 0; o >>= 1) val += __shfl_down_sync(0xffffffffu, val, o);
        if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = val;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        double acc = 0.0;
        for (int w = 0; w < EN_T / 32; ++w) acc += red[threadIdx.x][w];
        partial[blockIdx.x * 8 + threadIdx.x] = acc;
    }
}

void launch_energy(const double *x3, const double *v3, const double *m, long long n, double G, double eps2,
                   const int32_t *sys_off, int nsys, double *partial, int nblk, cudaStream_t s)
{
    if (n <= 0) return;
    const bool one = !(sys_off && nsys > 1), soft = eps2 != 0.0;
    const auto k = one ? (soft ? k_energy<true, true> : k_energy<true, false>)
                       : (soft ? k_energy<false, true> : k_energy<false, false>);
    k<<<nblk, EN_T, 0, s>>>(x3, v3, m, n, G, eps2, 1.0, sys_off, nsys, partial);
    CC_COUNT_LAUNCH(1);
}

}  // namespace cc

// ------------------------------------------------------------ peak probe
// FMA throughput microbenchmarks (the ALU roofline denominators): every
// thread advances 8 independent FMA chains; flops = 2 per FMA.
namespace cc {

template <typename T>
__global__ void __launch_bounds__(256) k_probe_fma(T b, T c, int iters, T *out)
{
    T a0 = (T)threadIdx.x, a1 = a0 + (T)1, a2 = a0 + (T)2, a3 = a0 + (T)3;
    T a4 = a0 + (T)4, a5 = a0 + (T)5, a6 = a0 + (T)6, a7 = a0 + (T)7;
    for (int i = 0; i < iters; ++i) {
        a0 = fma(a0, b, c); a1 = fma(a1, b, c); a2 = fma(a2, b, c); a3 = fma(a3, b, c);
        a4 = fma(a4, b, c); a5 = fma(a5, b, c); a6 = fma(a6, b, c); a7 = fma(a7, b, c);
    }
    const T r = ((a0 + a1) + (a2 + a3)) + ((a4 + a5) + (a6 + a7));
    if (r == (T)-12345.678) out[blockIdx.x] = r;  // keeps the chains live
}

double probe_fma(int fp64, int nsm, cudaStream_t s)
{
    const int blocks = nsm * 8, threads = 256;
    const int iters = fp64 ? 512 : 16384;
    void *out = nullptr;
    cudaMalloc(&out, blocks * 8);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    for (int rep = 0; rep < 4; ++rep) {
        cudaEventRecord(e0, s);
        if (fp64)
            k_probe_fma<double><<<blocks, threads, 0, s>>>(0.999999, 1e-7, iters, (double *)out);
        else
            k_probe_fma<float><<<blocks, threads, 0, s>>>(0.999999f, 1e-7f, iters, (float *)out);
        CC_COUNT_LAUNCH(1);
        cudaEventRecord(e1, s);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (rep > 0 && ms < best) best = ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    const double flops = 2.0 * 8.0 * (double)iters * blocks * threads;
    return flops / (best * 1e-3);
}

}  // namespace cc
