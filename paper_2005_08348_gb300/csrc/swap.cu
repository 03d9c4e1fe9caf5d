// Lipid-exchange trials (arXiv:2005.08348 Sec. 2, Eq. 1) and MDAS
// alchemical moves (Sec. 2, Eqs. 2-3) for sm_103a.
//
// An exchange swaps the lipid types of two lipids at fixed coordinates; its
// energy change is a sum over pairs with at least one bead whose type
// changes, of u(new types) - u(old types), evaluated in FP64 from exact
// integer separations.  Bonded terms do not depend on type and drop out.
//
// Batched trials keep sequential semantics: all pending trials are evaluated
// speculatively against the current types; a single thread then walks them in
// order and resolves every trial that no earlier accepted or still pending
// trial can influence (no shared lipid and no bead of one within reach of the
// other); the rest are re-evaluated in the next round.
#include <cmath>

#include "mdas_trial.cuh"

namespace mdas {

// Sum over the neighbours j in one of the 27 cells around changed bead i of
// u(new_i, new_j) - u(old_i, old_j); pairs of two changed beads are counted
// by the lower id only.  Candidates are culled in FP32 from exact integer
// separations (those within float rounding of rc are decided in FP64); the
// energies are FP64.  Types come from a functor of (meta, id) and a predicate
// telling whether a neighbour is changed.
template <class NewT, class Changed>
__device__ double bead_delta(const SysDev &S, const Params &P, int i, uint4 pi, int old_i, int new_i, int slot,
                             NewT newt, Changed changed) {
    const int nx = P.nc[0], ny = P.nc[1], nz = P.nc[2];
    const int cx = (int)(((unsigned long long)pi.x * (unsigned)nx) >> 32);
    const int cy = (int)(((unsigned long long)pi.y * (unsigned)ny) >> 32);
    const int cz = (int)(((unsigned long long)pi.z * (unsigned)nz) >> 32);
    const int dz = slot / 9 - 1, dy = (slot / 3) % 3 - 1, dx = slot % 3 - 1;
    const int x = (cx + dx + nx) % nx, y = (cy + dy + ny) % ny, z = (cz + dz + nz) % nz;
    const int cj = (z * ny + y) * nx + x;
    const int li = meta_lip(pi.w), ki = meta_k(pi.w);
    const uint32_t em = P.excl[ki];
    double acc = 0.0;
    const int e = cj * P.capc + S.cell_n[cj];
    for (int p = cj * P.capc; p < e; ++p) {
        const uint4 pj = __ldcg(&S.spos[p]);
        const int ix = (int)(pi.x - pj.x), iy = (int)(pi.y - pj.y), iz = (int)(pi.z - pj.z);
        const float fx = (float)ix * P.qsf[0], fy = (float)iy * P.qsf[1], fz = (float)iz * P.qsf[2];
        const float r2f = fx * fx + fy * fy + fz * fz;
        if (!(r2f < P.rc2f) || r2f == 0.0f) continue;
        const int j = S.sorted_id[p];
        if (j == i) continue;
        const bool chj = changed(pj.w, j);
        if (chj && j < i) continue;
        if (li >= 0 && meta_lip(pj.w) == li && ((em >> meta_k(pj.w)) & 1u)) continue;
        const double ex = (double)ix * P.qs[0], ey = (double)iy * P.qs[1], ez = (double)iz * P.qs[2];
        const double r2 = fma(ex, ex, fma(ey, ey, ez * ez));
        if (!inside_rc(P, r2, r2f)) continue;
        const int old_j = meta_ta(pj.w);
        const int new_j = chj ? newt(pj.w, j) : old_j;
        acc += pair_du(P, old_i, old_j, new_i, new_j, r2, r2f);
    }
    return acc;
}

// -------------------------------------------------------------- proposals
// grid (ceil(n/128), n_sys): trial t of system y draws (a, b, u) from
// Philox counter (0, trial + t, TAG_SWAP, 0); a, b by multiply-shift.
__global__ void k_swap_propose(const SysDev *__restrict__ sys, int n) {
    const SysDev &S = sys[blockIdx.y];
    const Params &P = *S.p;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const unsigned long long T = S.c->trial + (unsigned long long)t;
    const uint4 w = draw4(P, 0u, (uint32_t)T, TAG_SWAP, 0u);
    const int a = pick(w.x, P.n_lip), b = pick(w.y, P.n_lip);
    S.tprop[t] = make_int4(a, b, -1, -1);
    S.tu[t] = unit53(w.z, w.w);
    S.tstate[t] = 0;
    if (t == 0) S.c->pending = n;              // this system has trials to resolve
}

// bounding box of lipid l in fixed-point units: centre and half widths
__device__ void lipid_box(const SysDev &S, const Params &P, int l, int4 *cen, int4 *half) {
    const uint4 p0 = S.pos[l * P.bpl];
    int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
    for (int k = 1; k < P.bpl; ++k) {
        const uint4 pk = S.pos[l * P.bpl + k];
        const int d[3] = {(int)(pk.x - p0.x), (int)(pk.y - p0.y), (int)(pk.z - p0.z)};
        for (int e = 0; e < 3; ++e) { lo[e] = min(lo[e], d[e]); hi[e] = max(hi[e], d[e]); }
    }
    *cen = make_int4((int)(p0.x + (uint32_t)(int)(((long long)lo[0] + hi[0]) / 2)),
                     (int)(p0.y + (uint32_t)(int)(((long long)lo[1] + hi[1]) / 2)),
                     (int)(p0.z + (uint32_t)(int)(((long long)lo[2] + hi[2]) / 2)), 0);
    *half = make_int4((hi[0] - lo[0]) / 2 + 1, (hi[1] - lo[1]) / 2 + 1, (hi[2] - lo[2]) / 2 + 1, 0);
}

// grid (ceil(2n/128), n_sys): the boxes of both lipids of every trial
__global__ void k_swap_boxes(const SysDev *__restrict__ sys, int n) {
    const SysDev &S = sys[blockIdx.y];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 2 * n) return;
    const int4 pr = S.tprop[k >> 1];
    lipid_box(S, *S.p, (k & 1) ? pr.y : pr.x, &S.lbox[k], &S.lhalf[k]);
}

__device__ __forceinline__ bool boxes_near(const Params &P, int4 ca, int4 ha, int4 cb, int4 hb) {
    const long long gx = llabs((long long)(int)((uint32_t)ca.x - (uint32_t)cb.x)) - ha.x - hb.x;
    const long long gy = llabs((long long)(int)((uint32_t)ca.y - (uint32_t)cb.y)) - ha.y - hb.y;
    const long long gz = llabs((long long)(int)((uint32_t)ca.z - (uint32_t)cb.z)) - ha.z - hb.z;
    return gx < (long long)P.rcu[0] && gy < (long long)P.rcu[1] && gz < (long long)P.rcu[2];
}

// conflict bit (t, t') for t' < t: a shared lipid, or a lipid of one within
// reach of a lipid of the other.  grid (ceil(n*W/128), n_sys), W = words per row.
__global__ void k_swap_conflicts(const SysDev *__restrict__ sys, int n) {
    const SysDev &S = sys[blockIdx.y];
    const Params &P = *S.p;
    const int W = (n + 31) / 32;
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n * W) return;
    const int t = g / W, wd = g % W;
    const int4 pt = S.tprop[t];
    uint32_t bits = 0;
    for (int k = 0; k < 32; ++k) {
        const int u = wd * 32 + k;
        if (u >= t) break;
        const int4 pu = S.tprop[u];
        bool c = pt.x == pu.x || pt.x == pu.y || pt.y == pu.x || pt.y == pu.y;
        for (int s = 0; s < 2 && !c; ++s)
            for (int r = 0; r < 2 && !c; ++r)
                c = boxes_near(P, S.lbox[2 * t + s], S.lhalf[2 * t + s], S.lbox[2 * u + r], S.lhalf[2 * u + r]);
        if (c) bits |= 1u << k;
    }
    S.conflict[t * W + wd] = bits;
}

void launch_swap_propose(const LaunchCtx &L, int n) {
    dim3 g1((n + 127) / 128, L.n_sys);
    k_swap_propose<<<g1, 128, 0, L.stream>>>(L.sys, n);
    if (n > 1) {   // a single trial has no earlier trial to conflict with
        dim3 g0((2 * n + 127) / 128, L.n_sys);
        k_swap_boxes<<<g0, 128, 0, L.stream>>>(L.sys, n);
        const int W = (n + 31) / 32;
        dim3 g2((n * W + 127) / 128, L.n_sys);
        k_swap_conflicts<<<g2, 128, 0, L.stream>>>(L.sys, n);
    }
}

// ------------------------------------------------------------ speculation
// grid (n * 9, n_sys): CTA (t, g) sums the dE of trial t over the 3
// neighbour cells (dz, dy) = g of every changed bead (FP64, fixed-order
// reduction); the 9 partial sums are added in order by the resolve kernel.

__global__ void __launch_bounds__(128) k_swap_dE(const SysDev *__restrict__ sys, int n) {
    const SysDev &S = sys[blockIdx.y];
    const Params &P = *S.p;
    const int t = blockIdx.x / DE_GROUPS, grp = blockIdx.x % DE_GROUPS;
    __shared__ double sh[128];
    __shared__ int chg_id[2 * MAXT], chg_new[2 * MAXT], chg_old[2 * MAXT];
    __shared__ int nchg, kmask;
    if (S.tstate[t] != 0) return;
    const int4 pr = S.tprop[t];
    const int a = pr.x, b = pr.y;
    const int ta = S.ltype[a], tb = S.ltype[b];
    if (threadIdx.x == 0) {
        if (grp == 0) S.tprop[t] = make_int4(a, b, ta, tb);
        int m = 0, nc = 0;
        if (a != b && ta != tb) {
            for (int k = 0; k < P.bpl; ++k)
                if (P.lbt[ta * 16 + k] != P.lbt[tb * 16 + k]) m |= 1 << k;
            for (int side = 0; side < 2; ++side)
                for (int k = 0; k < P.bpl; ++k)
                    if ((m >> k) & 1) {
                        chg_id[nc] = (side ? b : a) * P.bpl + k;
                        chg_old[nc] = P.lbt[(side ? tb : ta) * 16 + k];
                        chg_new[nc] = P.lbt[(side ? ta : tb) * 16 + k];
                        ++nc;
                    }
        }
        nchg = nc;
        kmask = m;
    }
    __syncthreads();
    const int nc = nchg, m = kmask;
    auto changed = [&](uint32_t mj, int) {
        const int l = meta_lip(mj);
        return (l == a || l == b) && ((m >> meta_k(mj)) & 1);
    };
    auto newt = [&](uint32_t mj, int) {
        const int l = meta_lip(mj);
        return (int)P.lbt[(l == a ? tb : ta) * 16 + meta_k(mj)];
    };
    double acc = 0.0;
    for (int it = threadIdx.x; it < nc * 3; it += blockDim.x) {
        const int ci = it / 3, slot = grp * 3 + it % 3;
        const int i = chg_id[ci];
        acc += bead_delta(S, P, i, S.pos[i], chg_old[ci], chg_new[ci], slot, newt, changed);
    }
    const double s = block_sum(acc, sh);
    if (threadIdx.x == 0) S.tdE[t * DE_GROUPS + grp] = s;
}

void launch_swap_dE(const LaunchCtx &L, int n) {
    dim3 g(n * DE_GROUPS, L.n_sys);
    k_swap_dE<<<g, 128, 0, L.stream>>>(L.sys, n);
}

// New meta word of bead id: the id-ordered positions, and the list-ordered
// copy while the pair list is valid.
__device__ __forceinline__ void set_meta(const SysDev &S, const Params &P, int id, uint32_t m) {
    S.pos[id].w = m;
    const Counters &C = *S.c;
    if (!C.nl_stale) S.lpos[(size_t)C.nl_par * P.n + S.lk[id]].w = m;
}

// Rewrite the A type of every bead of lipid l for lipid type lt (position
// arrays and the cell-ordered copy).
__device__ void set_lipid_type(const SysDev &S, const Params &P, int l, int lt) {
    S.ltype[l] = lt;
    for (int k = 0; k < P.bpl; ++k) {
        const int id = l * P.bpl + k;
        const int bt = P.lbt[lt * 16 + k];
        const uint32_t m = meta_make(bt, bt, k, l + 1);
        set_meta(S, P, id, m);
        S.spos[S.sidx[id]].w = m;
    }
}


// One exchange trial per system from the pair list, after a step of the separate
// launches: grid (TRIAL_PARTS, n_sys).
template <int G>
__global__ void __launch_bounds__(GRP) k_trial_nl(const SysDev *__restrict__ sys) {
    __shared__ TrialSmem sm;
    const SysDev &S = sys[blockIdx.y];
    trial_nl_part<G>(S, blockIdx.x, S.c->nl_par, Grp{(int)threadIdx.x, 1}, sm, false);
}

void launch_trial_nl(const LaunchCtx &L) {
    dim3 g(TRIAL_PARTS, L.n_sys);
    if (L.lanes == 2) k_trial_nl<2><<<g, 128, 0, L.stream>>>(L.sys);
    else k_trial_nl<4><<<g, 128, 0, L.stream>>>(L.sys);
}


// one block per system, one thread walks the trials in order
__global__ void k_swap_resolve(const SysDev *__restrict__ sys, int n) {
    const SysDev &S = sys[blockIdx.x];
    const Params &P = *S.p;
    Counters &C = *S.c;
    if (threadIdx.x != 0) return;
    const int W = (n + 31) / 32;
    uint32_t blocked[MAX_ROUND_TRIALS / 32];
    for (int w = 0; w < W; ++w) blocked[w] = 0;
    int pending = 0;
    for (int t = 0; t < n; ++t) {
        if (S.tstate[t] != 0) continue;
        bool blk = false;
        for (int w = 0; w <= t / 32 && !blk; ++w) {
            uint32_t bits = S.conflict[t * W + w];
            if (w == t / 32) bits &= (1u << (t % 32)) - 1u;      // only earlier trials
            blk = (bits & blocked[w]) != 0;
        }
        if (blk) { blocked[t / 32] |= 1u << (t % 32); ++pending; continue; }
        const int4 pr = S.tprop[t];
        const int a = pr.x, b = pr.y;
        const double u = S.tu[t];
        TrialRec r;
        r.a = a; r.b = b; r.u = u; r.dE = 0.0; r.accepted = 0;
        r.index = C.trial + (unsigned long long)t;
        r.null_trial = (a == b) || (S.ltype[a] == S.ltype[b]);
        if (!r.null_trial) {
            double dE = 0.0;
            for (int g = 0; g < DE_GROUPS; ++g) dE += S.tdE[t * DE_GROUPS + g];
            r.dE = dE;
            if (r.dE + P.kT * log(u) <= 0.0) {
                const int ta = S.ltype[a], tb = S.ltype[b];
                set_lipid_type(S, P, a, tb);
                set_lipid_type(S, P, b, ta);
                r.accepted = 1;
                blocked[t / 32] |= 1u << (t % 32);
            }
        }
        S.log[r.index % LOG_CAP] = r;
        C.trials++;
        C.force_evals++;
        C.null_trials += r.null_trial;
        C.accepted += r.accepted;
        S.tstate[t] = 1;
    }
    // the trial counter advances once, in the round that resolves this
    // system's last trial (in a batch, later rounds for other systems'
    // trials find nothing pending here)
    if (C.pending != 0) {
        C.rounds++;
        if (pending == 0) C.trial += (unsigned long long)n;
    }
    C.pending = pending;
}

void launch_swap_resolve(const LaunchCtx &L, int n) {
    k_swap_resolve<<<L.n_sys, 32, 0, L.stream>>>(L.sys, n);
}

// ------------------------------------------------------------------ MDAS
// The pairs of an alchemical move: explicit (mode 1), drawn over all lipids
// (mode 0, Philox (j, move, TAG_MDAS_PAIR, 0) for candidate j), or drawn
// across the leaflets (mode 2, Philox (j, move, TAG_LEAFLET, 0); a candidate
// is kept when a lies in leaflet 0 and b in leaflet 1 by leaf[]).  Then the
// B types of the pairs' beads.
//
// One block per system: its first warp draws 32 candidates at a time and takes
// them in order, then every thread marks beads (one thread for all of it spent
// its time in some 400 dependent loads, 60 us for 8 pairs; a move of 6 pairs
// over 18 steps at 700 lipids takes 1018 us for 1053).
constexpr int MDAS_THREADS = 128;
static_assert(2 * MAX_PAIRS <= MDAS_THREADS, "a thread per lipid of the pairs");
__global__ void __launch_bounds__(MDAS_THREADS) k_mdas_select(const SysDev *__restrict__ sys, int n_pairs, int max_tries,
                                                              int mode, const int *__restrict__ leaf) {
    constexpr unsigned FULL = 0xffffffffu;
    const SysDev &S = sys[blockIdx.x];
    const Params &P = *S.p;
    Counters &C = *S.c;
    __shared__ int pairs[2 * MAX_PAIRS];
    __shared__ int n_sel;
    const int t = threadIdx.x, lane = t & 31;
    if (mode == 1) {
        if (t < 2 * C.n_pairs) pairs[t] = C.pairs[t];
        if (t == 0) n_sel = C.n_pairs;
    } else if (t < 32) {
        const uint32_t tag = mode == 2 ? TAG_LEAFLET : TAG_MDAS_PAIR;
        int np = 0;
        for (int j0 = 0; j0 < max_tries && np < n_pairs; j0 += 32) {
            const uint4 w = draw4(P, (uint32_t)(j0 + lane), (uint32_t)C.move, tag, 0u);
            const int a = pick(w.x, P.n_lip), b = pick(w.y, P.n_lip);
            bool ok = j0 + lane < max_tries && a != b && S.ltype[a] != S.ltype[b];
            if (mode == 2) ok = ok && leaf[a] == 0 && leaf[b] == 1;
            for (unsigned left = __ballot_sync(FULL, ok); left && np < n_pairs; left &= left - 1u) {
                const int src = __ffs(left) - 1;
                const int ca = __shfl_sync(FULL, a, src), cb = __shfl_sync(FULL, b, src);
                bool used = false;
                for (int k = lane; k < 2 * np; k += 32) used = used || pairs[k] == ca || pairs[k] == cb;
                if (__any_sync(FULL, used)) continue;
                if (lane == 0) { pairs[2 * np] = ca; pairs[2 * np + 1] = cb; }
                __syncwarp();
                ++np;
            }
        }
        for (int k = lane; k < 2 * np; k += 32) C.pairs[k] = pairs[k];
        if (lane == 0) C.n_pairs = n_sel = np;
    }
    __syncthreads();
    for (int x = t; x < 2 * n_sel * P.bpl; x += MDAS_THREADS) {
        const int y = x / P.bpl, k = x - y * P.bpl;          // lipid pairs[y] takes the type of its partner
        const int l = pairs[y], id = l * P.bpl + k;
        set_meta(S, P, id, meta_make(meta_ta(S.pos[id].w), P.lbt[S.ltype[pairs[y ^ 1]] * 16 + k], k, l + 1));
    }
    if (t == 0) C.w = 0.0;
}

void launch_mdas_select(const LaunchCtx &L, int n_pairs, int max_tries, int mode, const int *leaf) {
    k_mdas_select<<<L.n_sys, MDAS_THREADS, 0, L.stream>>>(L.sys, n_pairs, max_tries, mode, leaf);
}

// Leaflet of every lipid of system 0: 0 when its head (local index head_k)
// lies above its last bead, i.e. the z steps of its bonds from the head to
// the last bead, each at its minimum image, sum to a drop (exact integers).
__global__ void k_leaflets(const SysDev *__restrict__ sys, int head_k, int *__restrict__ leaf) {
    const SysDev &S = *sys;
    const Params &P = *S.p;
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= P.n_lip) return;
    long long drop = 0;
    for (int k = head_k; k < P.bpl - 1; ++k) {
        const int b = l * P.bpl + k;
        drop += (int)(S.pos[b].z - S.pos[b + 1].z);
    }
    leaf[l] = drop > 0 ? 0 : 1;
}

void launch_leaflets(const LaunchCtx &L, int n_lip, int head_k, int *leaf) {
    k_leaflets<<<(n_lip + 127) / 128, 128, 0, L.stream>>>(L.sys, head_k, leaf);
}

__global__ void k_mdas_set_lambda(const SysDev *__restrict__ sys, double lambda, int in_at) {
    const SysDev &S = sys[blockIdx.x];
    if (threadIdx.x == 0) { S.c->lambda = lambda; S.c->in_at = in_at; }
}

void launch_mdas_set_lambda(const LaunchCtx &L, double lambda, int in_at) {
    k_mdas_set_lambda<<<L.n_sys, 32, 0, L.stream>>>(L.sys, lambda, in_at);
}

// grid (2 * MAX_PAIRS, n_sys): CTA x handles lipid x of the pair list; the
// changed beads are those whose A and B types differ (U_B - U_A at the
// current coordinates, pairs of two changed beads counted once).
__global__ void __launch_bounds__(128) k_mdas_dE(const SysDev *__restrict__ sys, int n_lip) {
    const SysDev &S = sys[blockIdx.y];
    const Params &P = *S.p;
    Counters &C = *S.c;
    __shared__ double sh[128];
    const int x = blockIdx.x;
    if (x >= (n_lip >= 0 ? n_lip : 2 * C.n_pairs)) return;
    const int l = C.pairs[x];
    auto changed = [&](uint32_t mj, int) { return meta_ta(mj) != meta_tb(mj); };
    auto newt = [&](uint32_t mj, int) { return meta_tb(mj); };
    double acc = 0.0;
    for (int it = threadIdx.x; it < P.bpl * 27; it += blockDim.x) {
        const int k = it / 27, slot = it % 27;
        const int i = l * P.bpl + k;
        const uint4 pi = S.pos[i];
        if (meta_ta(pi.w) == meta_tb(pi.w)) continue;
        acc += bead_delta(S, P, i, pi, meta_ta(pi.w), meta_tb(pi.w), slot, newt, changed);
    }
    const double s = block_sum(acc, sh);
    if (threadIdx.x == 0) C.w_part[x] = s;
}

// The same sum from the pair list (valid right after an MD block), one block
// per lipid x: grid (2 * MAX_PAIRS, n_sys).
template <int G>
__global__ void __launch_bounds__(128) k_mdas_dE_nl(const SysDev *__restrict__ sys, double l0, double l1) {
    const SysDev &S = sys[blockIdx.y];
    __shared__ double sh[GRP / 32];
    const int x = blockIdx.x;
    if (x >= 2 * S.c->n_pairs) return;
    const double w = mdas_work_part<G>(S, x, S.c->nl_par, Grp{(int)threadIdx.x, 1}, sh, l0, l1);
    if (threadIdx.x == 0) S.c->w_part[x] = w;
}

// w += dlambda * (sum of the parts), or the sum itself when the parts hold
// the step's work already (soft-core path from the pair list, as_is)
__global__ void k_mdas_accumulate(const SysDev *__restrict__ sys, double dlambda, int n_lip, int as_is) {
    const SysDev &S = sys[blockIdx.x];
    Counters &C = *S.c;
    if (threadIdx.x != 0) return;
    const int to_result = n_lip >= 0;
    const int nl = to_result ? n_lip : 2 * C.n_pairs;
    double s = 0.0;
    for (int x = 0; x < nl; ++x) s += C.w_part[x];
    if (to_result) S.result[8] = s;
    else C.w += as_is && S.p->sc_delta > 0.0 ? s : dlambda * s;
}

void launch_mdas_dE_nl(const LaunchCtx &L, double l0, double l1, double dlambda) {
    dim3 g(2 * MAX_PAIRS, L.n_sys);
    if (L.lanes == 2) k_mdas_dE_nl<2><<<g, 128, 0, L.stream>>>(L.sys, l0, l1);
    else k_mdas_dE_nl<4><<<g, 128, 0, L.stream>>>(L.sys, l0, l1);
    k_mdas_accumulate<<<L.n_sys, 32, 0, L.stream>>>(L.sys, dlambda, -1, 1);
}

void launch_mdas_dE(const LaunchCtx &L, double dlambda) {
    dim3 g(2 * MAX_PAIRS, L.n_sys);
    k_mdas_dE<<<g, 128, 0, L.stream>>>(L.sys, -1);
    k_mdas_accumulate<<<L.n_sys, 32, 0, L.stream>>>(L.sys, dlambda, -1, 0);
}

// Eq. 3: accept with min(1, exp(-w/kT)), i.e. w + kT ln u <= 0, u from
// Philox (0, move, TAG_MDAS_ACC, 0) words 2-3.
__global__ void __launch_bounds__(MDAS_THREADS) k_mdas_accept(const SysDev *__restrict__ sys) {
    const SysDev &S = sys[blockIdx.x];
    const Params &P = *S.p;
    Counters &C = *S.c;
    __shared__ int newt[2 * MAX_PAIRS];
    __shared__ int accept;
    const int t = threadIdx.x, n = 2 * C.n_pairs;
    if (t == 0) {
        const uint4 w = draw4(P, 0u, (uint32_t)C.move, TAG_MDAS_ACC, 0u);
        const double u = unit53(w.z, w.w);
        accept = C.n_pairs > 0 && C.w + P.kT * log(u) <= 0.0;
        S.result[9] = u;
    }
    if (t < n) newt[t] = S.ltype[C.pairs[t ^ 1]];
    __syncthreads();
    if (accept) {
        if (t < n) S.ltype[C.pairs[t]] = newt[t];
        for (int x = t; x < n * P.bpl; x += MDAS_THREADS) {
            const int y = x / P.bpl, k = x - y * P.bpl, l = C.pairs[y];
            const int bt = P.lbt[newt[y] * 16 + k];
            set_meta(S, P, l * P.bpl + k, meta_make(bt, bt, k, l + 1));
        }
    }
    if (t == 0) {
        C.mdas_accept = accept;
        C.move++;
        C.moves++;
        C.moves_accepted += accept;
        C.in_at = 0;
        C.lambda = 0.0;
    }
}

void launch_mdas_accept(const LaunchCtx &L) { k_mdas_accept<<<L.n_sys, MDAS_THREADS, 0, L.stream>>>(L.sys); }

template <typename V4>
__global__ void k_restore(const SysDev *__restrict__ sys, const int2 *__restrict__ bmap) {
    const int2 bm = bmap[blockIdx.x];
    const SysDev &S = sys[bm.x];
    const int i = bm.y + threadIdx.x;
    if (i >= S.p->n || S.c->mdas_accept) return;
    if (i == 0) {   // the velocities go back to the snapshot, the positions leave the pair list
        S.c->ke_fresh = 0;
        S.c->ke_pending = 0;
        S.c->nl_stale = 1;
    }
    if (i < 4 * KE_SLOTS) (&S.c->ke_slot[0][0][0])[i] = 0;
    S.pos[i] = S.pos_snap[i];
    reinterpret_cast<V4 *>(S.vel)[i] = reinterpret_cast<const V4 *>(S.vel_snap)[i];
}

template <typename V4>
__global__ void k_snapshot(const SysDev *__restrict__ sys, const int2 *__restrict__ bmap) {
    const int2 bm = bmap[blockIdx.x];
    const SysDev &S = sys[bm.x];
    const int i = bm.y + threadIdx.x;
    if (i >= S.p->n) return;
    S.pos_snap[i] = S.pos[i];
    reinterpret_cast<V4 *>(S.vel_snap)[i] = reinterpret_cast<const V4 *>(S.vel)[i];
}

void launch_mdas_restore(const LaunchCtx &L) {
    if (L.precision == 1) k_restore<Dbl4><<<L.beads->n, BEAD_BLOCK, 0, L.stream>>>(L.sys, L.beads->d);
    else k_restore<float4><<<L.beads->n, BEAD_BLOCK, 0, L.stream>>>(L.sys, L.beads->d);
}

void launch_snapshot(const LaunchCtx &L) {
    if (L.precision == 1) k_snapshot<Dbl4><<<L.beads->n, BEAD_BLOCK, 0, L.stream>>>(L.sys, L.beads->d);
    else k_snapshot<float4><<<L.beads->n, BEAD_BLOCK, 0, L.stream>>>(L.sys, L.beads->d);
}

// Hypothetical collective type change: lipids C.pairs[0..n) get the types in
// C.pairs[MAX_PAIRS..MAX_PAIRS+n) as B types; dE = U_B - U_A into result[8];
// the B marks are removed again afterwards.
__global__ void __launch_bounds__(MDAS_THREADS) k_mark_b(const SysDev *__restrict__ sys, int n, int clear) {
    const SysDev &S = sys[blockIdx.x];
    const Params &P = *S.p;
    Counters &C = *S.c;
    for (int x = threadIdx.x; x < n * P.bpl; x += MDAS_THREADS) {
        const int y = x / P.bpl, k = x - y * P.bpl, l = C.pairs[y], id = l * P.bpl + k;
        const uint32_t m = S.pos[id].w;
        const int tb = clear ? meta_ta(m) : (int)P.lbt[C.pairs[MAX_PAIRS + y] * 16 + k];
        const uint32_t nm = meta_make(meta_ta(m), tb, k, l + 1);
        set_meta(S, P, id, nm);
        S.spos[S.sidx[id]].w = nm;
    }
}

void launch_delta_energy(const LaunchCtx &L, int n) {
    k_mark_b<<<L.n_sys, MDAS_THREADS, 0, L.stream>>>(L.sys, n, 0);
    dim3 g(2 * MAX_PAIRS, L.n_sys);
    k_mdas_dE<<<g, 128, 0, L.stream>>>(L.sys, n);
    k_mdas_accumulate<<<L.n_sys, 32, 0, L.stream>>>(L.sys, 0.0, n, 0);
    k_mark_b<<<L.n_sys, MDAS_THREADS, 0, L.stream>>>(L.sys, n, 1);
}

// ------------------------------------------- trials in order, many per launch
// Exchange trials over the pair lists (G list columns per bead) and semi-grand
// lipid mutations over the cells (G = 0; Sec. 2: a random lipid turned into a
// lipid of another type under a Metropolis test), with the result of processing
// them one after another.  Coordinates do not change, so what a trial's dE
// depends on are the types of its own lipids and of the lipids with a bead
// inside the cutoff of a changed bead.  A chunk of trials runs as
//   k_chain_propose: who draws which lipid (per lipid a list of the chunk's
//     trials);
//   k_chain_eval: every trial's dE against the types the chunk starts with, a
//     block per trial, and as it walks the partners the earlier trials of the
//     chunk whose acceptance would change it (a bit per trial);
//   k_chain_walk: one cluster of blocks per system decides the trials in order;
//     one whose bits meet an accepted trial is evaluated again, by the whole
//     cluster (the FP64 pair terms bound a single SM: some 1300 of them for an
//     exchange at 28 operations, two per clock).
// dE is one fixed sum of CHAIN_SLOTS slots, whichever kernel computes it, so
// the records do not depend on the chunks.
//
// Measured, a call of 256 trials: exchanges on a 1424-lipid bilayer 530 to 630 us
// by state and session (a launch per trial: 2580), mutations on a 4608-lipid
// bilayer 350 to 435 us (one block for all of them: 10970); the same call again
// and again on one state 473 and 281 us.
//
// Mutation trial T draws Philox (0, T, TAG_MUTATE, 0): lipid a from word 0, the
// new type among the other n_lt - 1 types from word 1, u from words 2-3; accept
// iff dE - (mu[new] - mu[old]) + kT ln u <= 0.
constexpr int CHAIN_BLOCKS = 8;                // blocks of a cluster of k_chain_walk
constexpr int CHAIN_THREADS = 128;
constexpr int CHAIN_SLOTS = CHAIN_BLOCKS * CHAIN_THREADS;
constexpr int CHAIN_SUMS = CHAIN_SLOTS / 32;   // warp sums of one dE
constexpr int CHAIN_WORDS = CHAIN_MAX / 32;

struct ChainProp {
    int a, b;                                  // the lipids (a mutation has a alone: b = a)
    uint32_t w1;                               // mutation: the word that picks the new type
    double u;
};

template <int G>
__device__ __forceinline__ ChainProp chain_draw(const Params &P, unsigned long long T) {
    const uint4 w = draw4(P, 0u, (uint32_t)T, G ? TAG_SWAP : TAG_MUTATE, 0u);
    ChainProp r;
    r.a = pick(w.x, P.n_lip);
    r.b = G ? pick(w.y, P.n_lip) : r.a;
    r.w1 = w.y;
    r.u = unit53(w.z, w.w);
    return r;
}

// The trial's two types, the current ones of a and b or a's old and new one,
// and its changed beads, into sm; by one warp.
template <int G>
__device__ __forceinline__ void chain_setup(const SysDev &S, const ChainProp &pr, const uint4 *cur, int lane, TrialSmem &sm) {
    const Params &P = *S.p;
    const int ta = __ldcg(&S.ltype[pr.a]);
    if constexpr (G > 0) {
        trial_beads<G>(S, pr.a, pr.b, ta, __ldcg(&S.ltype[pr.b]), cur, lane, sm, [](int) {});
    } else {
        const int tn = P.n_lt > 1 ? (ta + 1 + pick(pr.w1, P.n_lt - 1)) % P.n_lt : ta;
        const int oi = lane < P.bpl ? P.lbt[ta * 16 + lane] : 0, ni = lane < P.bpl ? P.lbt[tn * 16 + lane] : 0;
        const unsigned bal = __ballot_sync(0xffffffffu, oi != ni);
        if (oi != ni) {
            const int o = __popc(bal & ((1u << lane) - 1u)), id = pr.a * P.bpl + lane;
            sm.chg_id[o] = id;
            sm.chg_pos[o] = S.pos[id];
            sm.chg_old[o] = oi;
            sm.chg_new[o] = ni;
        }
        if (lane == 0) {
            sm.nchg = __popc(bal);
            sm.ta = ta;
            sm.tb = tn;
        }
    }
}

// One lane's part of the dE of the trial in sm: the warp's entries are those of
// slots slot0 .. slot0 + 31, of every CHAIN_SLOTS.  An exchange's entry is a list
// entry of a changed bead; a mutation's is every fourth bead of one of a changed
// bead's 27 cells.  ring: 64 entries of this warp.
//
// The FP64 pipe (two operations per clock and SM, whole warps) bounds it, and
// less than half of a list's entries and a sixth of the cells' beads are inside
// the cutoff: the warp culls in FP32, lets the survivors wait in the ring and
// takes 32 at a time through FP64, and it fetches four rounds of entries at a
// time: 256 exchange trials at 1424 lipids 13% less, 256 mutation trials at 4608
// lipids 20% less than each lane with its own entries, one after another.
template <int G, class Near>
__device__ __forceinline__ double chain_warp(const SysDev &S, const ChainProp &pr, const uint4 *cur, const TrialSmem &sm,
                                             int slot0, int lane, int4 *ring, Near near) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int ROUNDS = 4;
    const Params &P = *S.p;
    const float q0 = P.qsf[0], q1 = P.qsf[1], q2 = P.qsf[2];
    double acc = 0.0;
    int head = 0, tail = 0;
    auto take = [&](int nt) {
        if (lane < nt) {
            const int4 e = ring[(head + lane) & 63];
            const double ex = (double)e.x * P.qs[0], ey = (double)e.y * P.qs[1], ez = (double)e.z * P.qs[2];
            const float fx = (float)e.x * q0, fy = (float)e.y * q1, fz = (float)e.z * q2;
            const double r2 = fma(ex, ex, fma(ey, ey, ez * ez));
            const float r2f = fx * fx + fy * fy + fz * fz;
            if (inside_rc(P, r2, r2f))
                acc += pair_du(P, e.w & 15, (e.w >> 4) & 15, (e.w >> 8) & 15, (e.w >> 12) & 15, r2, r2f);
        }
        head += nt;
        __syncwarp();
    };
    // a candidate pj (v: there is one) of bead pi; types(): its old and new
    // types, or a negative number when the pair does not count
    auto offer = [&](bool v, uint4 pi, uint4 pj, auto types) {
        const int ix = (int)(pi.x - pj.x), iy = (int)(pi.y - pj.y), iz = (int)(pi.z - pj.z);
        const float fx = (float)ix * q0, fy = (float)iy * q1, fz = (float)iz * q2;
        const float r2f = fx * fx + fy * fy + fz * fz;
        int ty = -1;
        if (v && r2f < P.rc2f && r2f != 0.0f) ty = types();
        const unsigned bal = __ballot_sync(FULL, ty >= 0);
        if (ty >= 0) ring[(tail + __popc(bal & ((1u << lane) - 1u))) & 63] = make_int4(ix, iy, iz, ty);
        tail += __popc(bal);
        __syncwarp();
        if (tail - head >= 32) take(32);
    };
    if constexpr (G > 0) {
        const int a = pr.a, b = pr.b, cols = sm.nchg * G, total = sm.it_beg[cols];
        for (int f0 = slot0; f0 < total; f0 += ROUNDS * CHAIN_SLOTS) {
            int ci[ROUNDS], kj[ROUNDS];
            uint4 pj[ROUNDS];
#pragma unroll
            for (int u = 0; u < ROUNDS; ++u) {
                const int f = f0 + u * CHAIN_SLOTS + lane;
                int lo = 0, hi = cols - 1;        // the (bead, column) holding entry f
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (sm.it_beg[mid] <= f) lo = mid; else hi = mid - 1;
                }
                ci[u] = lo / G;
                kj[u] = f < total ? S.nl[nl_at<G>(P.npad, sm.chg_k[ci[u]], f - sm.it_beg[lo], lo % G)] : -1;
            }
#pragma unroll
            for (int u = 0; u < ROUNDS; ++u)
                pj[u] = kj[u] >= 0 ? __ldcg(cur + MDAS_IDX(*S.c, kj[u], P.n)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < ROUNDS; ++u) {
                if (f0 + u * CHAIN_SLOTS >= total) break;
                const int c = ci[u];
                offer(kj[u] >= 0, sm.chg_pos[c], pj[u], [&]() {
                    const int l = meta_lip(pj[u].w), k = meta_k(pj[u].w);
                    near(l);
                    const bool ch = (l == a || l == b) && ((sm.m >> k) & 1);
                    if (ch && l * P.bpl + k < sm.chg_id[c]) return -1;     // a changed pair once, by the lower id
                    const int oj = meta_ta(pj[u].w);
                    const int nj = ch ? (int)P.lbt[(l == a ? sm.tb : sm.ta) * 16 + k] : oj;
                    return sm.chg_old[c] | oj << 4 | sm.chg_new[c] << 8 | nj << 12;
                });
            }
        }
    } else {
        const int a = pr.a, ta = sm.ta, tn = sm.tb, total = sm.nchg * 27 * 4;
        const int nx = P.nc[0], ny = P.nc[1], nz = P.nc[2];
        for (int f0 = slot0; f0 < total; f0 += CHAIN_SLOTS) {
            const int f = f0 + lane, ci = f < total ? f / 108 : 0, q = f % 108, o = q >> 2;
            const uint4 pi = sm.chg_pos[ci];
            int x = (int)(((unsigned long long)pi.x * (unsigned)nx) >> 32) + o % 3 - 1;
            int y = (int)(((unsigned long long)pi.y * (unsigned)ny) >> 32) + (o / 3) % 3 - 1;
            int z = (int)(((unsigned long long)pi.z * (unsigned)nz) >> 32) + o / 9 - 1;
            x += x < 0 ? nx : (x >= nx ? -nx : 0);
            y += y < 0 ? ny : (y >= ny ? -ny : 0);
            z += z < 0 ? nz : (z >= nz ? -nz : 0);
            const int cj = (z * ny + y) * nx + x, e = f < total ? S.cell_n[cj] : 0, i = sm.chg_id[ci];
            const int ki = meta_k(pi.w);
            const uint32_t em = P.excl[ki];
            const uint4 *sp = S.spos + (size_t)cj * P.capc;
            for (int p0 = q & 3; __any_sync(FULL, p0 < e); p0 += 4 * ROUNDS) {
                uint4 pj[ROUNDS];
#pragma unroll
                for (int u = 0; u < ROUNDS; ++u)
                    pj[u] = p0 + 4 * u < e ? __ldcg(sp + p0 + 4 * u) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int u = 0; u < ROUNDS; ++u) {
                    if (!__any_sync(FULL, p0 + 4 * u < e)) break;
                    offer(p0 + 4 * u < e, pi, pj[u], [&]() {
                        const int l = meta_lip(pj[u].w), k = meta_k(pj[u].w);
                        if (l == a && k == ki) return -1;                  // the bead itself
                        near(l);
                        const int old = meta_ta(pj[u].w);
                        const int nj = l == a ? (int)P.lbt[tn * 16 + k] : old;
                        const bool ch = l == a && P.lbt[ta * 16 + k] != P.lbt[tn * 16 + k];
                        if (ch && l * P.bpl + k < i) return -1;            // a changed pair once, by the lower id
                        if (l == a && ((em >> k) & 1u)) return -1;         // bonded
                        return sm.chg_old[ci] | old << 4 | sm.chg_new[ci] << 8 | (ch ? nj : old) << 12;
                    });
                }
            }
        }
    }
    if (tail != head) take(tail - head);
    return acc;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;                                  // lane 0
}

// The sum of the warp sums, on every lane of a warp (a fixed tree: one after
// another they took as long as the cutoff tests).
__device__ __forceinline__ double chain_total(const double *sums, int lane) {
    static_assert(CHAIN_SUMS == 32, "a warp sum per lane");
    double v = sums[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// grid (1, n_sys): node 2 t + side + 1 of trial t enters the list of the lipid
// it draws (0: the end; the walk empties the lists again)
template <int G>
__global__ void __launch_bounds__(CHAIN_MAX) k_chain_propose(const SysDev *__restrict__ sys, int m) {
    const SysDev &S = sys[blockIdx.y];
    const int t = threadIdx.x;
    if (t >= m) return;
    const ChainProp pr = chain_draw<G>(*S.p, S.c->trial + (unsigned long long)t);
    for (int side = 0; side < (G ? 2 : 1); ++side)
        S.tnext[2 * t + side] = atomicExch(&S.thead[side ? pr.b : pr.a], 2 * t + side + 1);
}

// grid (m, n_sys)
template <int G>
__global__ void __launch_bounds__(CHAIN_THREADS) k_chain_eval(const SysDev *__restrict__ sys) {
    const SysDev &S = sys[blockIdx.y];
    const Params &P = *S.p;
    __shared__ TrialSmem sm;
    __shared__ double sums[CHAIN_SUMS];
    __shared__ int4 ring[CHAIN_THREADS / 32][64];
    __shared__ unsigned bits[CHAIN_WORDS];
    const int t = blockIdx.x, x = threadIdx.x, lane = x & 31;
    const ChainProp pr = chain_draw<G>(P, S.c->trial + (unsigned long long)t);
    const uint4 *cur = S.lpos + (size_t)S.c->nl_par * P.n;
    if (x < CHAIN_WORDS) bits[x] = 0u;
    if (x < 32) chain_setup<G>(S, pr, cur, lane, sm);
    __syncthreads();
    // the earlier trials that draw lipid l
    auto meets = [&](int l) {
        if (l < 0) return;
        for (int node = S.thead[l]; node; node = S.tnext[node - 1]) {
            const int u = (node - 1) >> 1;
            if (u < t) atomicOr(&bits[u >> 5], 1u << (u & 31));
        }
    };
    if (x < 2) meets(x ? pr.b : pr.a);
    for (int i = 0; i < CHAIN_BLOCKS; ++i) {
        const double s = warp_sum(chain_warp<G>(S, pr, cur, sm, CHAIN_THREADS * i + (x & ~31), lane, ring[x >> 5], meets));
        if (lane == 0) sums[(CHAIN_THREADS / 32) * i + (x >> 5)] = s;
    }
    __syncthreads();
    if (x < CHAIN_WORDS) S.conflict[t * CHAIN_WORDS + x] = bits[x];
    if (x < 32) {
        const double dE = chain_total(sums, lane);
        if (lane == 0) {
            S.tdE[t] = dE;
            S.tprop[t] = make_int4(pr.a, pr.b, sm.ta, sm.tb);
        }
    }
}

__device__ __forceinline__ unsigned cluster_addr(const void *p, unsigned rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
// (not the .aligned forms: those want the whole warp to arrive together, and
// the code before it diverges by lane)
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// grid (CHAIN_BLOCKS, n_sys), one cluster per system: trials 0 .. m - 1 of the
// chunk in order.  spec: k_chain_eval has run (else every trial is evaluated
// here).  The first warp of the first block decides; for a trial that needs
// its dE it hands the cluster the trial's number and takes back the warp sums.
template <int G>
__global__ void __cluster_dims__(CHAIN_BLOCKS, 1, 1) __launch_bounds__(CHAIN_THREADS)
k_chain_walk(const SysDev *__restrict__ sys, int m, int spec) {
    const SysDev &S = sys[blockIdx.y];
    const Params &P = *S.p;
    Counters &C = *S.c;
    __shared__ TrialSmem sm;
    __shared__ double sums[CHAIN_SUMS];
    __shared__ int4 ring[CHAIN_THREADS / 32][64];
    __shared__ int cmd;
    __shared__ unsigned bits[CHAIN_MAX * CHAIN_WORDS];
    const int x = threadIdx.x, lane = x & 31;
    const unsigned rank = blockIdx.x;
    const bool lead = rank == 0 && x < 32;
    const unsigned long long T0 = C.trial;
    const uint4 *cur = S.lpos + (size_t)C.nl_par * P.n;
    const bool lists = !C.nl_stale;
    if (spec && rank == 0)
        for (int i = x; i < m * CHAIN_WORDS; i += CHAIN_THREADS) bits[i] = S.conflict[i];
    __syncthreads();
    // the leading warp: the next trial, the accepted ones (lane w: word w),
    // counts; 32 trials' proposals and dE at a time, one per lane
    int t = 0, n_null = 0, n_acc = 0;
    unsigned accepted = 0u;
    bool fresh = false;                        // sums hold the dE of trial t
    ChainProp mine;
    double mine_dE = 0.0;
    int mine_ta = 0, mine_tb = 0;
    for (;;) {
        if (lead) {
            int next = -1;
            for (; t < m; ++t) {
                if ((t & 31) == 0 && !fresh) {
                    mine = chain_draw<G>(P, T0 + (unsigned long long)min(t + lane, m - 1));
                    if (spec && t + lane < m) {
                        mine_dE = S.tdE[t + lane];
                        const int4 q = S.tprop[t + lane];
                        mine_ta = q.z;
                        mine_tb = q.w;
                    }
                }
                const unsigned hit = spec && lane < CHAIN_WORDS ? bits[t * CHAIN_WORDS + lane] & accepted : 0u;
                if (!fresh && (!spec || __any_sync(0xffffffffu, hit != 0u))) {
                    next = t;
                    break;
                }
                const int src = t & 31;
                TrialRec r;
                r.a = __shfl_sync(0xffffffffu, mine.a, src);
                const int b = __shfl_sync(0xffffffffu, mine.b, src);
                r.u = __shfl_sync(0xffffffffu, mine.u, src);
                double dE = __shfl_sync(0xffffffffu, mine_dE, src);
                int ta = __shfl_sync(0xffffffffu, mine_ta, src), tb = __shfl_sync(0xffffffffu, mine_tb, src);
                if (fresh) {
                    dE = chain_total(sums, lane);
                    ta = sm.ta;
                    tb = sm.tb;
                    fresh = false;
                }
                r.b = G ? b : tb;
                r.index = T0 + (unsigned long long)t;
                r.null_trial = (G && r.a == b) || ta == tb;
                r.dE = r.null_trial ? 0.0 : dE;
                r.accepted = !r.null_trial && metropolis(G ? dE : dE - (C.mu[tb] - C.mu[ta]), P.kT, r.u);
                n_null += r.null_trial;
                n_acc += r.accepted;
                if (lane == 0) S.log[r.index % LOG_CAP] = r;
                if (r.accepted) {
                    // the new types, one bead per lane
                    const int side = lane >= P.bpl, k = side ? lane - P.bpl : lane;
                    if (lane < (G ? 2 : 1) * P.bpl) {
                        const int l = side ? b : r.a, id = l * P.bpl + k;
                        const int bt = P.lbt[(side ? ta : tb) * 16 + k];
                        const uint32_t mm = meta_make(bt, bt, k, l + 1);
                        S.pos[id].w = mm;
                        if (lists) const_cast<uint4 *>(cur)[S.lk[id]].w = mm;
                        if (!G) S.spos[S.sidx[id]].w = mm;
                    }
                    if (lane == 0) {
                        S.ltype[r.a] = tb;
                        if (G) S.ltype[b] = ta;
                    }
                    if (lane == (t >> 5)) accepted |= 1u << (t & 31);
                }
            }
            if (lane == 0) cmd = next;
        }
        cluster_sync();
        int todo;
        asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(todo) : "r"(cluster_addr(&cmd, 0)) : "memory");
        if (todo < 0) break;
        const ChainProp pr = chain_draw<G>(P, T0 + (unsigned long long)todo);
        if (x < 32) chain_setup<G>(S, pr, cur, lane, sm);
        __syncthreads();
        const double s = warp_sum(chain_warp<G>(S, pr, cur, sm, CHAIN_THREADS * rank + (x & ~31), lane, ring[x >> 5],
                                                [](int) {}));
        if (lane == 0)
            asm volatile("st.shared::cluster.f64 [%0], %1;"
                         :: "r"(cluster_addr(&sums[(CHAIN_THREADS / 32) * rank + (x >> 5)], 0)), "d"(s) : "memory");
        cluster_sync();
        fresh = true;
    }
    cluster_sync();                            // every block has read the last number
    if (lead && lane == 0) {
        C.trials += m;
        C.force_evals += m;
        C.null_trials += n_null;
        C.accepted += n_acc;
        C.pending = 0;
        C.trial = T0 + (unsigned long long)m;
    }
    if (spec && rank == 0)
        for (int i = x; i < m; i += CHAIN_THREADS) {
            const ChainProp pr = chain_draw<G>(P, T0 + (unsigned long long)i);
            S.thead[pr.a] = 0;
            S.thead[pr.b] = 0;
        }
}

// A chunk is long enough to fill the GPU with evaluations and short enough that
// few of its trials meet an accepted one: a trial of a bilayer of n_lip lipids
// has some 25 lipids in reach, so a chunk of n_lip / 16 evaluates about one
// trial in five again.  From CHAIN_MIN trials on (shorter chunks of small
// bilayers, where most trials meet, are walked without the first evaluation).
// Returns the number of launches.
template <int G>
static int chain_launch(const LaunchCtx &L, int n, int max_lip) {
    int launches = 0;
    const int chunk = max_lip / 16 >= CHAIN_MAX ? CHAIN_MAX : max_lip / 16;
    const int spec = chunk >= CHAIN_MIN && n >= CHAIN_MIN;
    const int step = spec ? chunk : CHAIN_MAX;
    for (int done = 0; done < n; done += step) {
        const int m = n - done < step ? n - done : step;
        launches += spec ? 3 : 1;
        if (spec) {
            k_chain_propose<G><<<dim3(1, L.n_sys), CHAIN_MAX, 0, L.stream>>>(L.sys, m);
            k_chain_eval<G><<<dim3(m, L.n_sys), CHAIN_THREADS, 0, L.stream>>>(L.sys);
        }
        k_chain_walk<G><<<dim3(CHAIN_BLOCKS, L.n_sys), CHAIN_THREADS, 0, L.stream>>>(L.sys, m, spec);
    }
    return launches;
}

void launch_swap_trials(const LaunchCtx &L, int n, int max_lip) {
    if (L.lanes == 2) chain_launch<2>(L, n, max_lip);
    else chain_launch<4>(L, n, max_lip);
}

int launch_mutation_trials(const LaunchCtx &L, int n, int max_lip) { return chain_launch<0>(L, n, max_lip); }

// ----------------------------------------------------------------- Philox
__global__ void k_philox(uint32_t k0, uint32_t k1, uint32_t c1, uint32_t c2, uint32_t c3, int n, uint4 *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = philox4x32_10(make_uint4((uint32_t)i, c1, c2, c3), k0, k1);
}

void launch_philox(uint32_t k0, uint32_t k1, uint32_t c1, uint32_t c2, uint32_t c3, int n, uint4 *out, cudaStream_t st) {
    k_philox<<<(n + 255) / 256, 256, 0, st>>>(k0, k1, c1, c2, c3, n, out);
}

}  // namespace mdas
