// Checklist walk and local expansions (Sec. 3.1).
//
// Sink cells are walked top-down, one tree level per launch.  A warp (on a level of few sinks, a
// block) owns one sink cell k and its checklist: the sources its parent left on the checklist ("remain on the
// checklist for further consideration by the children of the sink cell") plus, for the
// root, the root itself.  Each lane takes one entry, evaluates the opening criterion and
// the warp or block appends the entry to one of five places with ballot/popc ranks:
//   accept  -> k's local-expansion list (CC for a cell, CP for a particle)
//   defer   -> the checklist handed to k's children
//   PC, PP  -> the group's interaction lists (k a group: <= g particles)
//   open    -> its two children, or for a bucket its particles with R_O = 0, are
//              appended to k's own queue and examined in turn.
// The criterion (single precision, fixed operation order, no fused multiply-add):
//   d = |com_k - com_s|, R_O = b_max / theta (0 for a particle or a one-particle cell)
//   accept if d > 1.5 R_O(k) + R_O(s) and the bounding boxes are >= 2 eps apart
//   k not a group: defer if s is point-like or R_O(s) <= R_O(k), else open
//   k a group:     PP if s is point-like; PC if d > R_O(s) + b_max(k); PP if s is a
//                  bucket; else open.
// Outputs are staged in per-warp scratch and copied to contiguous per-cell ranges, so each
// cell's lists are in a deterministic order whatever the scheduling.
//
// The local expansion of a walked cell is L_k = L2L(L_parent) + sum of M2L (CC) and P2L
// (CP) terms.  The M2L and P2L terms and the top-down passes follow the walk's last level.  A level's
// local lists are complete when its walk kernel ends, so they can also run level by level beside the
// walk (walk_levels).
#include <limits.h>

#include <algorithm>

#include "expansions.cuh"
#include "fmm_internal.cuh"
#include "mlp.cuh"

#define WALK_WPB 4
#define WALK_THREADS (WALK_WPB * 32)

// Learned criterion (MODE 1): the pairs the network must decide wait in a list of the sink's until
// its queue runs dry.  They are then evaluated 32 per warp, which fills two tensor-core tiles, and
// return to the queue in the order they were met, marked with their decision; the next steps sort
// them like any other entry.  So the order of the queue does not depend on how many entries a step
// takes.  Marks: bit 30 accepted, bit 29 rejected (cell entries of an isolated box, whose indices
// stay below 2^29).
#define WALK_NET_ACC (1u << 30)
#define WALK_NET_REJ (1u << 29)

__device__ __forceinline__ float d2_ordered(float dx, float dy, float dz)
{
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

__device__ __forceinline__ float gap_axis(float lo_s, float hi_s, float lo_k, float hi_k)
{
    float g1 = __fsub_rn(lo_s, hi_k), g2 = __fsub_rn(lo_k, hi_s);
    float g = g1 > g2 ? g1 : g2;
    return g > 0.0f ? g : 0.0f;
}

// Resident blocks per SM the fixed-theta walk is compiled for: 6 (80 registers, all of the grid's 24
// warps per SM resident) against 5, walk phase 3.04 against 3.08 ms on the 128^3 NFW box and 15.5
// against 16.1 ms on a 256^3 box with a tenth of its particles active.
#ifndef FMM_WALK_MINB
#define FMM_WALK_MINB 6
#endif
// A level of fewer than FMM_WALK_TEAM_SINKS sinks per block of the grid gives every sink a whole
// block (walk_sinks).  Walk phase by this line, 128^3 NFW box / 200^3 box with the learned
// criterion: 1: 3.54 / 11.8 ms, 2: 3.21 / 11.8, 4: 3.08 / 11.7, 8: 3.11 / 11.7, 16: 3.23 / 11.8,
// every level: 3.22 / 13.9.
#ifndef FMM_WALK_TEAM_SINKS
#define FMM_WALK_TEAM_SINKS 4
#endif

// A large walk keeps every level's sinks in tree order (left before right, so in space): a sink then
// leaves its children in its own place, and two small kernels count and place them (k_front_count,
// k_front_place).  In the order in which the sinks before them happened to finish, neighbours drift
// apart level by level, and their sources, which they share, come from DRAM again each time.  The two
// launches per level cost a small walk more than the locality gives it.  Whole solve without / with the
// order, by cells: 128^3 NFW box (0.4 million) 7.81 / 8.21 ms, Plummer 6.3 million particles (1.13) 19.83 /
// 20.07, 12.7 million (2.28) 40.88 / 40.97, NFW 12.7 million (2.31) 41.8 / 42.2, 14.3 million (2.61) 47.4 / 47.4,
// 16.8 million (3.08) 56.7 / 56.6, Plummer 24 million (4.3) 71.7 / 71.5, a substep of it with a tenth active
// 43.6 / 42.8, 32 million (5.8) 96.9 / 96.3; in buckets of 8 and 4 the lines cross between 3 and 5 million.
// The learned criterion's longer queues gain earlier: Plummer 4.2 million particles (0.76) 15.96 / 15.59,
// 8 million (1.44) 28.8 / 28.1, 16.8 million (3.03) 55.4 / 54.2; NFW 4.2 million (0.78) 17.06 / 17.14, 6.3 million
// (1.15) 24.31 / 24.25, 8 million (1.47) 29.9 / 30.1, 16.8 million (3.08) 61.6 / 60.9.
#ifndef FMM_ORDER_CELLS
#define FMM_ORDER_CELLS (5LL << 19)
#endif
#ifndef FMM_ORDER_CELLS_NET
#define FMM_ORDER_CELLS_NET (1LL << 20)
#endif
#define FRONT_BITS 30  // of a frontier entry's length; above them, in an ordered walk, its children
#define FRONT_TILE FMM_FRONT_TILE

// What a walk level reads and writes (one kernel parameter).
struct WalkIO {
    const WalkNode* node;
    const float4* posf;
    const int* cnact;
    const int* f_cell;
    unsigned long long* f_cloff;
    int* f_cllen;
    bool ordered;  // sinks leave their children to k_front_place
    const unsigned int* cl_cur;
    int* f_cell_next;
    unsigned long long* f_cloff_next;
    int* f_cllen_next;
    unsigned int* cl_next;
    unsigned long long *lcc_off, *lcp_off;
    int *lcc_len, *lcp_len, *wcells;
    unsigned int *pp, *pc, *cc, *cp;
    int *cc_sink, *cp_sink;
    Group* groups;
    unsigned int* scratch;
    DevCounters* ctr;
    long long cap_front, cap_cl, cap_pp, cap_pc, cap_cc, cap_cp, cap_groups, cap_scr;
    int level, group;
    float four_eps2;
    // learned criterion and audit
    const float4* mnorm;
    const float* amin;
    float eps, band_lo, band_hi, tau, margin;
    const unsigned char* mlp_packed;
    int2* audit_pairs;
    long long audit_cap;
    const unsigned char* nogroup;
    PeriodicArgs pa;
};

// A team's shared words: the counts of every warp's step (two steps' worth), and broadcasts.
struct WalkShared {
    uint2 cnt[2][WALK_WPB];
    unsigned int srcpp;
    unsigned long long fi, at[5];
};

// Barrier of the TEAM warps that share a sink: the warp itself, or the whole block.
template <int TEAM>
__device__ __forceinline__ void team_sync()
{
    if (TEAM == 1) __syncwarp();
    else __syncthreads();
}

// A source as the criterion sees it: a cell's node, or a particle as a node of no extent.  A
// source in a periodic copy has its centre and box shifted in FP64, then rounded, read from the
// tables of those values (the axes with a non-zero shift).
template <bool PER>
__device__ __forceinline__ WalkNode walk_source(const WalkIO& w, unsigned int e, unsigned int q0, int ib)
{
    const unsigned int j = entry_index(e, ib);
    const bool part = (e & FMM_PARTICLE_BIT) != 0u;
    WalkNode S;
    const float4* src = part ? w.posf + j : reinterpret_cast<const float4*>(w.node + j);
    S.a = __ldg(src);
    if (!part) {
        S.b = __ldg(src + 1);
        S.c = __ldg(src + 2);
        S.d = __ldg(reinterpret_cast<const int4*>(src + 3));
    } else {
        S.d = make_int4(-1, -1, 0, 1);
    }
    if (PER && entry_copy(e, ib) != q0) {
        int nv[3];
        copy_shift(entry_copy(e, ib), w.pa.R, nv[0], nv[1], nv[2]);
        const int w2 = 2 * w.pa.R;
#pragma unroll
        for (int ax = 0; ax < 3; ax++) {
            if (nv[ax] == 0) continue;
            const long long slot = ((long long)j * 3 + ax) * w2 + shift_slot(nv[ax], w.pa.R);
            float4 g;
            if (part) g.x = w.pa.pshift[slot];
            else g = w.pa.cshift[slot];
            if (ax == 0) {
                S.a.x = g.x;
                S.b.x = g.y;
                S.c.x = g.z;
            } else if (ax == 1) {
                S.a.y = g.x;
                S.b.y = g.y;
                S.c.y = g.z;
            } else {
                S.a.z = g.x;
                S.b.z = g.y;
                S.c.z = g.z;
            }
        }
    }
    if (part) {
        S.a.w = 0.0f;
        S.b = S.c = S.a;
    }
    return S;
}

// The sinks of one level.  TEAM warps share a sink (1: every warp has its own; WALK_WPB: the whole
// block) and examine 32 * TEAM entries of its queue per step, one per lane.  Outcomes are ranked in
// queue order (ballots within a warp, the warps' counts through shared memory), so the lists and
// the queue come out in the same order whatever TEAM is.
//
// A step is a chain of a few hundred dependent instructions and two dependent loads (the entry, its
// node), 1.4 us with one warp per sink; a level lasts as long as its longest sink's chain of steps
// (up to 170 on the 128^3 NFW box) unless its sinks fill the GPU.  So a level of few sinks takes
// TEAM = WALK_WPB, which cuts every chain by that factor, and a full level takes TEAM = 1, which has
// no barriers and wastes fewer lanes on the ends of queues.  Walk phase with local expansions, one
// warp per sink on every level against this: 4.38 to 3.04 ms on the 128^3 NFW box, 2.04 to 1.24 ms
// on a 63^3 one, 0.49 to 0.37 ms on a 4096-particle box, 2.55 to 1.31 ms on a dual-tree substep.
//
// MODE 0: fixed-theta criterion.  MODE 1: learned criterion for source cells (the network
// decides inside the band, see mlp.cuh).  MODE 2: fixed criterion, and every (sink, source cell)
// pair of the band is recorded for labelling (audit).  PER: a periodic box (list entries carry a
// copy code above their index bits); the isolated walk is compiled without the decoding.
template <int MODE, bool PER, int TEAM>
__device__ __forceinline__ void walk_sinks(const WalkIO& w, const unsigned long long n_front,
                                           const unsigned long long wbase, WalkShared& sh,
                                           const unsigned char* walk_smem, unsigned char* mlp_scratch)
{
    constexpr int WIN = 32 * TEAM;
    const unsigned int q0 = PER ? copy_centre(w.pa.R) : 0u;
    const int ib = PER ? w.pa.ib : 31;  // index bits of a list entry
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int tl = TEAM == 1 ? lane : (int)threadIdx.x;  // position in the team
    const int tw = TEAM == 1 ? 0 : wl;                   // warp of the team
    const int cap = (int)min(w.cap_scr * TEAM, (long long)INT_MAX);
    DevCounters* const ctr = w.ctr;
    // the team's scratch: queue, deferred, accepted (multipole sources from the front, point sources
    // from the back), PP and PC entries; pairs for the network wait in the list that the sink leaves
    // unused (a group defers nothing, any other sink has no PP entries)
    unsigned int* const Q = w.scratch + ((long long)blockIdx.x * WALK_WPB + (TEAM == 1 ? wl : 0)) * 5 * w.cap_scr;
    unsigned int* const D = Q + w.cap_scr * TEAM;
    unsigned int* const A = D + w.cap_scr * TEAM;
    unsigned int* const P = A + w.cap_scr * TEAM;
    unsigned int* const C = P + w.cap_scr * TEAM;
    const unsigned int lt = fmm_lanemask_lt();
    unsigned long long w_entries = 0, n_mlp = 0;  // this team's statistics, added once at the end
    int w_max = 0;

    for (;;) {
        unsigned long long fi = 0;
        if (TEAM == 1) {
            if (lane == 0) fi = atomicAdd(&ctr->lv_work[w.level], 1ull);
            fi = __shfl_sync(FMM_FULL_MASK, fi, 0);
        } else {
            __syncthreads();  // the last sink's shared words are done with
            if (threadIdx.x == 0) {
                sh.fi = atomicAdd(&ctr->lv_work[w.level], 1ull);
                sh.srcpp = 0u;
            }
            __syncthreads();
            fi = sh.fi;
        }
        if (fi >= n_front) break;
        const int k = w.f_cell[fi];
        if (tl == 0 && (long long)(wbase + fi) < w.cap_front) w.wcells[wbase + fi] = k;
        const WalkNode K = w.node[k];
        // a group holds <= g particles; in a graded tree (dual trees) it is also no larger than the
        // fixed tree's groups around it
        const bool kg = K.d.w <= w.group && !(w.nogroup && w.nogroup[k]);
        const float rk = K.a.w, bk = K.b.w, rk15 = __fmul_rn(1.5f, rk);
        const float ak = MODE == 1 ? w.amin[k] : 0.0f, la = MODE == 1 ? mlp_log_accel(ak) : 0.0f;
        const unsigned int* const cl = w.cl_cur + w.f_cloff[fi];
        const int ncl = w.f_cllen[fi];
        unsigned int* const X = kg ? C : D;  // a group's PC entries, any other sink's deferred ones
        unsigned int* const W = kg ? D : P;  // pairs for the network (MODE 1)
        int total = ncl, na = 0, nap = 0, nx = 0, npp = 0, nw = 0;
        int base = 0, par = 0;
        int srcpp = 0;  // this lane's PP source particles
        bool overflow = false;
        for (;;) {
            while (base < total) {
                const int vi = base + tl;
                bool valid = vi < total;
                unsigned int e = 0u;
                if (valid) e = vi < ncl ? cl[vi] : Q[vi - ncl];
                base = min(base + WIN, total);  // entries appended by this step follow
                unsigned int decided = 0u;  // learned criterion: the network's decision carried by the entry
                if (MODE == 1 && !(e & FMM_PARTICLE_BIT)) {
                    decided = e & (WALK_NET_ACC | WALK_NET_REJ);
                    e &= ~(WALK_NET_ACC | WALK_NET_REJ);
                }
                bool acc = false, ptl = false, mid = false, pp = false, open = false, need = false;
                int4 sd = make_int4(-1, -1, 0, 0);
                if (valid) {
                    const WalkNode S = walk_source<PER>(w, e, q0, ib);
                    const float ro = S.a.w;
                    sd = S.d;
                    ptl = sd.w == 1;
                    const float d2 = d2_ordered(__fsub_rn(K.a.x, S.a.x), __fsub_rn(K.a.y, S.a.y), __fsub_rn(K.a.z, S.a.z));
                    const float thr = __fadd_rn(rk15, ro);
                    const float gap2 = d2_ordered(gap_axis(S.b.x, S.c.x, K.b.x, K.c.x),
                                                  gap_axis(S.b.y, S.c.y, K.b.y, K.c.y),
                                                  gap_axis(S.b.z, S.c.z, K.b.z, K.c.z));
                    acc = d2 > __fmul_rn(thr, thr) && gap2 >= w.four_eps2;
                    if (MODE != 0 && !ptl) {
                        float te;
                        int band = mlp_band(K, S, d2, gap2, w.four_eps2, w.band_lo, w.band_hi, te);
                        if (MODE == 1) {
                            if (band == 3 && decided) {
                                band = decided == WALK_NET_ACC ? 1 : 2;  // the network has decided
                            } else if (band == 3 && !(ak > 0.0f)) {
                                band = acc ? 1 : 2;  // no acceleration estimate: the fixed criterion decides
                            } else if (band == 3) {
                                float f[MLP_F];
                                mlp_pair_features(K, S, w.mnorm[entry_index(e, ib)], la, w.eps, f);
                                band = mlp_surrogate(reinterpret_cast<const float*>(walk_smem + MLPP_SUR), f, te, w.tau,
                                                     w.margin);
                            }
                            acc = band == 1;
                            need = band == 3;
                        } else if (band == 3) {
                            const unsigned long long q = atomicAdd(&ctr->n_audit, 1ull);
                            if ((long long)q < w.audit_cap) w.audit_pairs[q] = make_int2(k, (int)e);
                        }
                    }
                    // a pair for the network gives no output until it has been decided
                    if (MODE == 1 && need) {
                        valid = false;
                    } else if (!acc) {
                        if (!kg) {
                            mid = ptl || ro <= rk;  // defer
                            open = !mid;
                        } else if (ptl) {
                            pp = true;
                        } else {
                            const float u = __fadd_rn(ro, bk);
                            mid = d2 > __fmul_rn(u, u);  // PC
                            pp = !mid && sd.x < 0;       // a leaf (bucket) has no children
                            open = !mid && !pp;
                        }
                    }
                }
                // this warp's outcomes, in queue order
                const bool leaf = sd.x < 0;
                const unsigned int mA = __ballot_sync(FMM_FULL_MASK, acc && !ptl);
                const unsigned int mAp = __ballot_sync(FMM_FULL_MASK, acc && ptl);
                const unsigned int mX = __ballot_sync(FMM_FULL_MASK, mid);
                // a group opens no leaf; any other sink has no PP entries
                const unsigned int mP = __ballot_sync(FMM_FULL_MASK, kg ? pp : (open && leaf));
                const unsigned int mO = __ballot_sync(FMM_FULL_MASK, open && !leaf);
                const unsigned int mW = MODE == 1 ? __ballot_sync(FMM_FULL_MASK, need) : 0u;
                int qat = 2 * __popc(mO & lt), qtot = 2 * __popc(mO);
                if (!kg && mP) {
                    // leaves add 1 to 16 entries each: their counts bit by bit
                    const unsigned int c = open && leaf ? (unsigned int)sd.w : 0u;
#pragma unroll
                    for (int b = 0; b < 5; b++) {
                        const unsigned int m = __ballot_sync(FMM_FULL_MASK, (c >> b) & 1u);
                        qat += __popc(m & lt) << b;
                        qtot += __popc(m) << b;
                    }
                }
                int oA = na + __popc(mA & lt), oAp = nap + __popc(mAp & lt), oX = nx + __popc(mX & lt),
                    oP = npp + __popc(mP & lt), oW = MODE == 1 ? nw + __popc(mW & lt) : 0;
                qat += total - ncl;
                int tA = __popc(mA), tAp = __popc(mAp), tX = __popc(mX), tP = kg ? __popc(mP) : 0,
                    tW = MODE == 1 ? __popc(mW) : 0, tQ = qtot;
                if (TEAM > 1) {
                    // the counts of the team's warps: four of 8 bits (at most 32 * TEAM = 128 each), then
                    // the network's of 8 bits and the queue's (at most 512 * TEAM)
                    static_assert(WIN <= 255, "packed step counts");
                    if (lane == 0)
                        sh.cnt[par][wl] = make_uint2((unsigned)tA | (unsigned)tAp << 8 | (unsigned)tX << 16 | (unsigned)tP << 24,
                                                     (unsigned)tQ | (unsigned)tW << 24);
                    __syncthreads();
                    uint2 before = make_uint2(0u, 0u), all = make_uint2(0u, 0u);
#pragma unroll
                    for (int v = 0; v < TEAM; v++) {
                        const uint2 c = sh.cnt[par][v];
                        if (v == tw) before = all;
                        all.x += c.x;
                        all.y += c.y;
                    }
                    oA += before.x & 255u;
                    oAp += (before.x >> 8) & 255u;
                    oX += (before.x >> 16) & 255u;
                    oP += before.x >> 24;
                    qat += before.y & 0xffffffu;
                    tA = all.x & 255u;
                    tAp = (all.x >> 8) & 255u;
                    tX = (all.x >> 16) & 255u;
                    tP = all.x >> 24;
                    tQ = all.y & 0xffffffu;
                    if (MODE == 1) {
                        oW += before.y >> 24;
                        tW = all.y >> 24;
                    }
                    par ^= 1;
                }
                if (na + nap + tA + tAp > cap || nx + tX > cap || npp + tP > cap || total - ncl + tQ > cap ||
                    (MODE == 1 && nw + tW > cap)) {
                    overflow = true;
                    break;
                }
                if (acc) {
                    if (ptl) A[cap - 1 - oAp] = e;
                    else A[oA] = e;
                }
                if (mid) X[oX] = e;
                if (pp) {
                    P[oP] = e;
                    srcpp += sd.w;
                }
                if (MODE == 1 && need) W[oW] = e;
                // the children of opened cells, and the particles of opened leaves, stay in the source's copy
                const unsigned int qb = PER ? entry_copy(e, ib) << ib : 0u;
                if (open && !leaf) {
                    Q[qat] = (unsigned int)sd.x | qb;
                    Q[qat + 1] = (unsigned int)sd.y | qb;
                }
                if (!kg) {
                    // one opened leaf at a time, its particles along the lanes
                    for (unsigned int m = mP; m; m &= m - 1) {
                        const int src = __ffs(m) - 1;
                        const int at = __shfl_sync(FMM_FULL_MASK, qat, src), n = __shfl_sync(FMM_FULL_MASK, sd.w, src);
                        const unsigned int v = __shfl_sync(FMM_FULL_MASK, (unsigned int)sd.z | qb, src);
                        if (lane < n) Q[at + lane] = (v + (unsigned int)lane) | FMM_PARTICLE_BIT;
                    }
                }
                const int seen = total;
                na += tA;
                nap += tAp;
                nx += tX;
                npp += tP;
                nw += tW;
                total += tQ;
                // the next step's entries must be in place: a team's barrier is needed only when it reads
                // what this step appended (what earlier steps appended lies behind this step's barrier)
                if (TEAM == 1 || min(base + WIN, total) > seen) team_sync<TEAM>();
            }
            if (MODE == 0 || MODE == 2 || overflow || nw == 0) break;
            // the queue is dry: the network decides the waiting pairs, 32 per warp and turn
            if (total - ncl + nw > cap) {
                overflow = true;
                break;
            }
            team_sync<TEAM>();
            for (int b = tw * 32; b < nw; b += WIN) {
                const int cnt = min(32, nw - b);
                float f[MLP_F];
#pragma unroll
                for (int q = 0; q < MLP_F; q++) f[q] = 0.0f;
                unsigned int pe = 0u;
                if (lane < cnt) {
                    pe = W[b + lane];
                    const unsigned int j = entry_index(pe, ib);
                    mlp_pair_features(K, w.node[j], w.mnorm[j], la, w.eps, f);
                }
                const float pred = mlp_predict_warp(walk_smem, mlp_scratch, f, lane,
                                                    cnt == 32 ? FMM_FULL_MASK : (1u << cnt) - 1u);
                if (lane < cnt) Q[total - ncl + b + lane] = pe | (pred < w.tau ? WALK_NET_ACC : WALK_NET_REJ);
            }
            base = total;
            total += nw;
            n_mlp += (unsigned long long)nw;
            nw = 0;
            team_sync<TEAM>();
        }
        if (overflow) {
            if (tl == 0) atomicOr(&ctr->overflow, 1u);
            continue;
        }
        w_entries += (unsigned long long)total;
        w_max = max(w_max, total);
        // Room in the sink's lists: multipole sources (M2L) and point sources (P2L), and a group's PP and
        // PC entries or any other sink's checklist for its children, each in queue order.  One lane per
        // counter, so the atomics are in flight together.
        if (TEAM > 1 && kg) {
            srcpp = (int)__reduce_add_sync(FMM_FULL_MASK, (unsigned int)srcpp);
            if (lane == 0 && srcpp) atomicAdd(&sh.srcpp, (unsigned int)srcpp);
        }
        unsigned long long at = 0;
        if (tl < 5) {
            unsigned long long* c = tl == 0   ? &ctr->cc_len
                                    : tl == 1 ? &ctr->cp_len
                                    : tl == 2 ? (kg ? &ctr->pp_len : &ctr->lv_cl[w.level + 1])
                                    : tl == 3 ? &ctr->pc_len
                                              : &ctr->n_groups;
            const unsigned long long v = tl == 0 ? na : tl == 1 ? nap : tl == 2 ? (kg ? npp : nx) : tl == 3 ? nx : 1;
            if ((kg || tl < 3) && v) at = atomicAdd(c, v);
            if (TEAM > 1) sh.at[tl] = at;
        } else if (tl < 7) {  // the level's own counts
            const unsigned long long v = tl == 5 ? na : nap;
            if (v) atomicAdd(tl == 5 ? &ctr->lv_cc[w.level] : &ctr->lv_cp[w.level], v);
        }
        unsigned long long off, offp, xo, co, gi;
        if (TEAM == 1) {
            off = __shfl_sync(FMM_FULL_MASK, at, 0);
            offp = __shfl_sync(FMM_FULL_MASK, at, 1);
            xo = __shfl_sync(FMM_FULL_MASK, at, 2);
            co = __shfl_sync(FMM_FULL_MASK, at, 3);
            gi = __shfl_sync(FMM_FULL_MASK, at, 4);
        } else {
            __syncthreads();
            off = sh.at[0];
            offp = sh.at[1];
            xo = sh.at[2];
            co = sh.at[3];
            gi = sh.at[4];
        }
        bool fits = (long long)(off + na) <= w.cap_cc && (long long)(offp + nap) <= w.cap_cp;
        if (kg) fits = fits && (long long)(xo + npp) <= w.cap_pp && (long long)(co + nx) <= w.cap_pc && (long long)gi < w.cap_groups;
        else fits = fits && (long long)(xo + nx) <= w.cap_cl;
        if (!fits) {
            if (tl == 0) atomicOr(&ctr->overflow, 1u);
            continue;
        }
        for (int i = tl; i < na; i += WIN) {
            w.cc[off + i] = A[i];
            w.cc_sink[off + i] = k;
        }
        for (int i = tl; i < nap; i += WIN) {
            w.cp[offp + i] = A[cap - 1 - i];
            w.cp_sink[offp + i] = k;
        }
        if (tl == 0) {
            w.lcc_off[k] = off;
            w.lcc_len[k] = na;
            w.lcp_off[k] = offp;
            w.lcp_len[k] = nap;
        }
        if (kg) {
            if (TEAM == 1) srcpp = (int)__reduce_add_sync(FMM_FULL_MASK, (unsigned int)srcpp);
            else srcpp = (int)sh.srcpp;
            for (int i = tl; i < npp; i += WIN) w.pp[xo + i] = P[i];
            for (int i = tl; i < nx; i += WIN) w.pc[co + i] = C[i];
            if (tl == 0) {
                Group g;
                g.cell = k;
                g.first = K.d.z;
                g.count = K.d.w;
                g.pp_src = srcpp;
                g.pp_off = xo;
                g.pc_off = co;
                g.pp_len = npp;
                g.pc_len = nx;
                g.level = w.level;
                w.groups[gi] = g;
            }
        } else {
            for (int i = tl; i < nx; i += WIN) w.cl_next[xo + i] = D[i];
            if (w.ordered) {
                // over the sink's own entry, which has been read: its children's checklist, and which of them
                // hold active particles
                if (tl == 0) {
                    const unsigned int both = (w.cnact[K.d.x] > 0 ? 1u : 0u) | (w.cnact[K.d.y] > 0 ? 2u : 0u);
                    w.f_cloff[fi] = xo;
                    w.f_cllen[fi] = (int)((unsigned int)nx | both << FRONT_BITS);
                }
            } else if (tl < 2) {
                const int c = tl == 0 ? K.d.x : K.d.y;
                if (w.cnact[c] > 0) {
                    const unsigned long long fj = atomicAdd(&ctr->lv_front[w.level + 1], 1ull);
                    if ((long long)fj < w.cap_front) {
                        w.f_cell_next[fj] = c;
                        w.f_cloff_next[fj] = xo;
                        w.f_cllen_next[fj] = nx;
                    } else {
                        atomicOr(&ctr->overflow, 1u);
                    }
                }
            }
        }
    }
    if (tl == 0) {
        if (MODE == 1 && n_mlp) atomicAdd(&ctr->n_mlp, n_mlp);
        if (w_entries) {
            atomicAdd(&ctr->lv_entries[w.level], w_entries);
            atomicMax(&ctr->lv_max_entries[w.level], (unsigned long long)w_max);
        }
    }
}

template <int MODE, bool PER>
__global__ void __launch_bounds__(WALK_THREADS, MODE == 1 ? 4 : FMM_WALK_MINB) k_walk_level(const __grid_constant__ WalkIO w)
{
    __shared__ WalkShared sh;
    extern __shared__ __align__(16) unsigned char walk_smem[];
    DevCounters* const ctr = w.ctr;
    const unsigned long long n_front = *(volatile unsigned long long*)&ctr->lv_front[w.level];
    // this level's sinks go to the walked-cell list after the levels before it
    const unsigned long long wbase = *(volatile unsigned long long*)&ctr->lv_base[w.level];
    if (blockIdx.x == 0 && threadIdx.x == 0) ctr->lv_base[w.level + 1] = wbase + n_front;
    const bool team = n_front < (unsigned long long)gridDim.x * FMM_WALK_TEAM_SINKS;
    if ((unsigned long long)blockIdx.x * (team ? 1 : WALK_WPB) >= n_front) return;  // no sink is left for this block
    if (MODE == 1) {
        mlp_load_smem(w.mlp_packed, walk_smem);
        __syncthreads();
    }
    unsigned char* mlp_scratch = walk_smem + MLPP_SIZE + (threadIdx.x >> 5) * MLP_WARP_SCRATCH;
    if (team) walk_sinks<MODE, PER, WALK_WPB>(w, n_front, wbase, sh, walk_smem, mlp_scratch);
    else walk_sinks<MODE, PER, 1>(w, n_front, wbase, sh, walk_smem, mlp_scratch);
}

// Children per tile of a level's sinks.
__global__ void __launch_bounds__(FRONT_TILE) k_front_count(int level, long long cap, const int* __restrict__ f_cllen,
                                                           unsigned int* __restrict__ part,
                                                           const DevCounters* __restrict__ ctr)
{
    __shared__ unsigned int sum;
    const long long n = min((long long)ctr->lv_front[level], cap);
    for (long long t = blockIdx.x; t * FRONT_TILE < n; t += gridDim.x) {
        const long long i = t * FRONT_TILE + threadIdx.x;
        if (threadIdx.x == 0) sum = 0u;
        __syncthreads();
        const unsigned int c = __reduce_add_sync(FMM_FULL_MASK, i < n ? __popc((unsigned int)f_cllen[i] >> FRONT_BITS) : 0);
        if ((threadIdx.x & 31) == 0 && c) atomicAdd(&sum, c);
        __syncthreads();
        if (threadIdx.x == 0) part[t] = sum;
    }
}

// The next level's sinks in the order of their parents, from the tiles' counts.
__global__ void __launch_bounds__(FRONT_TILE) k_front_place(int level, const WalkNode* __restrict__ node,
                                                           const int* __restrict__ f_cell,
                                                           const unsigned long long* __restrict__ f_cloff,
                                                           const int* __restrict__ f_cllen, int* __restrict__ cell_next,
                                                           unsigned long long* __restrict__ cloff_next,
                                                           int* __restrict__ cllen_next, long long cap,
                                                           const unsigned int* __restrict__ part, DevCounters* __restrict__ ctr)
{
    __shared__ unsigned long long before;
    __shared__ unsigned int warp[FRONT_TILE / 32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const long long n = min((long long)ctr->lv_front[level], cap);
    for (long long t = blockIdx.x; t * FRONT_TILE < n; t += gridDim.x) {
        if (tid == 0) before = 0ull;
        __syncthreads();
        unsigned int p = 0u;
        for (long long q = tid; q < t; q += FRONT_TILE) p += part[q];
        p = __reduce_add_sync(FMM_FULL_MASK, p);
        if (lane == 0 && p) atomicAdd(&before, (unsigned long long)p);
        const long long i = t * FRONT_TILE + tid;
        const unsigned int e = i < n ? (unsigned int)f_cllen[i] : 0u;
        const unsigned int c = __popc(e >> FRONT_BITS);
        unsigned int at = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int v = __shfl_up_sync(FMM_FULL_MASK, at, o);
            if (lane >= o) at += v;
        }
        if (lane == 31) warp[w] = at;
        __syncthreads();
        if (w == 0) {
            unsigned int v = warp[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int u = __shfl_up_sync(FMM_FULL_MASK, v, o);
                if (lane >= o) v += u;
            }
            warp[lane] = v;
        }
        __syncthreads();
        long long to = (long long)before + (w ? warp[w - 1] : 0u) + at - c;
        if (c) {
            const int4 d = node[f_cell[i]].d;
            const unsigned long long off = f_cloff[i];
            for (int h = 0; h < 2; h++) {
                if (!(e >> (FRONT_BITS + h) & 1u)) continue;
                if (to < cap) {
                    cell_next[to] = h ? d.y : d.x;
                    cloff_next[to] = off;
                    cllen_next[to] = (int)(e & ((1u << FRONT_BITS) - 1u));
                } else {
                    atomicOr(&ctr->overflow, 1u);
                }
                to++;
            }
        }
        if (tid == 0 && (t + 1) * FRONT_TILE >= n) ctr->lv_front[level + 1] = before + warp[FRONT_TILE / 32 - 1];
        __syncthreads();
    }
}

#define LOCAL_WPB 2
#define LOCAL_THREADS (LOCAL_WPB * 32)

// Own local expansions over the flat list of all local entries (every walked sink's CC and CP
// entries, contiguous per sink).  A warp takes ranges of the list, moved to the next sink boundaries so
// that no sink is split between warps, and walks each in chunks of 32, one entry per lane, so lanes
// stay busy whatever the list lengths.  Each sink's 56 coefficients are
// added strictly in list order (runs of equal sink along the lanes, a run that continues into
// the next chunk carried on): the result depends only on the sink's own list, not on where the
// list lies in the flat array or which warp took it.
//
// A range is about a sixteenth of a warp's share of the list, so that the last turn's idle warps cost
// little, but at least 64 entries (every range ends in a part-filled chunk; short lists then still
// reach all SMs) and at most 8192.  Walk phase with ranges of 512 whatever the list, against this: 384^3
// box 42.5 to 41.4 ms, 256^3 substep 14.0 to 13.5, 128^3 2.74 to 2.62, 4096 particles 0.31 to 0.265.
#define LF_TURNS 16
#define LF_MAX 8192
#define LF_MIN 64

// Centres enter as float pairs (cen_diff): the sink's (hk, lk), a cell's from cen, a particle's
// from posf (hi, and its mass) and plo (lo); a source in a periodic copy has its pair shifted
// (cen_shift) by the copy's integer offset.
__device__ __forceinline__ void local_offset(unsigned int e, const float4& hk, const float4& lk, float4& hs, float4& ls,
                                             int ib, int R, float& rx, float& ry, float& rz)
{
    const unsigned int q = entry_copy(e, ib);
    if (q != copy_centre(R)) {
        int nx, ny, nz;
        copy_shift(q, R, nx, ny, nz);
        cen_shift(hs.x, ls.x, (float)nx);
        cen_shift(hs.y, ls.y, (float)ny);
        cen_shift(hs.z, ls.z, (float)nz);
    }
    rx = cen_diff(hk.x, lk.x, hs.x, ls.x);
    ry = cen_diff(hk.y, lk.y, hs.y, ls.y);
    rz = cen_diff(hk.z, lk.z, hs.z, ls.z);
}

// M2L sources of a chunk in shared memory, a row each: the moments, then the centre pair.  Read by a
// lane per source, a warp's load would touch 32 lines; copied 16 bytes per lane along the records it
// touches 8 (16 for the centres), and the copies need no registers, so the next chunk's are in flight
// while this one's sources are evaluated.  Walk phase with this, and with a sink's end known from the
// next chunk's first sink instead of two more dependent loads: 384^3 box 40.2 to 38.5 ms, batch of 27
// million particles 12.3 to 11.5, 256^3 substep 13.4 to 13.1, 128^3 NFW box 2.63 to 2.59; smaller
// boxes take the same time.  L1 prefetches of the next sinks' centres gave nothing more.
#define M2L_ROW (FMM_NMOM + 12)  // floats: a multiple of 4 that is 4 or 12 mod 16 keeps a quarter warp's reads apart
static_assert(FMM_NMOM == 32 && M2L_ROW % 4 == 0 && M2L_ROW % 8 != 0, "rows of 16-byte pieces");

__device__ __forceinline__ void copy16_async(float* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned int)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// entries e of the lanes below cnt
__device__ __forceinline__ void m2l_stage(unsigned int e, int cnt, const float4* __restrict__ cen,
                                          const float* __restrict__ rec, int ib, float* row, int lane)
{
    const unsigned int j = entry_index(e, ib);
#pragma unroll
    for (int q = 0; q < 8; q++) {
        const int s = q * 4 + (lane >> 3);
        const unsigned int js = __shfl_sync(FMM_FULL_MASK, j, s);
        if (s < cnt) copy16_async(row + s * M2L_ROW + (lane & 7) * 4, rec + (long long)js * FMM_NREC + (lane & 7) * 4);
    }
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const int s = q * 16 + (lane >> 1);
        const unsigned int js = __shfl_sync(FMM_FULL_MASK, j, s);
        if (s < cnt) copy16_async(row + s * M2L_ROW + FMM_NMOM + (lane & 1) * 4, cen + 2 * (long long)js + (lane & 1));
    }
}

// first entry of the first sink that starts at or after position p of the flat list
__device__ __forceinline__ long long local_boundary(long long p, long long total, const int* __restrict__ cc_sink,
                                                    const unsigned long long* __restrict__ lcc_off,
                                                    const int* __restrict__ lcc_len)
{
    if (p >= total) return total;
    const int k = cc_sink[p];
    const long long f = (long long)lcc_off[k];
    return f == p ? p : f + lcc_len[k];
}

// Two launches, one per list: KIND 0 the multipole sources (M2L), which write each sink's sum;
// KIND 1 the point sources (P2L), which add theirs to it (or write it, for a sink with no
// multipole source).  Every warp of a launch runs one kind of interaction.
// One level's entries: those of the sinks of walk level `level`, [sum of the earlier levels' counts,
// plus this level's), all of them complete when the level's walk kernel has ended; level -1: all.
#ifndef FMM_LOCAL_MINB
#define FMM_LOCAL_MINB 8  // resident blocks per SM the local-expansion kernels are compiled for (128 registers)
#endif
template <int KIND>
__global__ void __launch_bounds__(LOCAL_THREADS, FMM_LOCAL_MINB) k_local_flat(
    const unsigned int* __restrict__ cc, const int* __restrict__ cc_sink, const unsigned long long* __restrict__ lcc_off,
    const int* __restrict__ lcc_len, const int* __restrict__ lm2l_len, const float4* __restrict__ cen,
    const float4* __restrict__ posf, const float4* __restrict__ plo,
    const float* __restrict__ rec, float* __restrict__ Lown, long long cap_cc,
    float eps2, int ib, int R, int level, DevCounters* __restrict__ ctr)
{
    __shared__ float red[LOCAL_WPB][32][FMM_NL + 1];
    __shared__ __align__(16) float stage[KIND == 0 ? LOCAL_WPB : 1][KIND == 0 ? 32 * M2L_ROW : 4];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    float* const row = KIND == 0 ? stage[wl] : nullptr;  // M2L: this warp's staged sources
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    if (fmm_overflowed(ctr)) return;
    long long start = 0, total;
    if (level < 0) {  // every level's entries
        total = min((long long)*(volatile unsigned long long*)(KIND == 0 ? &ctr->cc_len : &ctr->cp_len), cap_cc);
    } else {
        const unsigned long long* lv = KIND == 0 ? ctr->lv_cc : ctr->lv_cp;
        for (int l = 0; l < level; l++) start += (long long)__ldcg(lv + l);
        total = min(start + (long long)__ldcg(lv + level), cap_cc);
    }
    if (start >= total) return;
    // ranges of whole chunks, about LF_TURNS per warp
    const long long len = min((long long)LF_MAX, max((long long)LF_MIN, (total - start) / (nw * LF_TURNS) / 32 * 32));
    const long long nranges = fmm_ceil_div(total - start, len);
    const int c0 = lane, c1 = lane + 32;  // this lane's coefficients in the reduction
    int nent = 0;
    for (long long r = gw; r < nranges; r += nw) {
        const long long r0 = local_boundary(start + r * len, total, cc_sink, lcc_off, lcc_len);
        const long long r1 = local_boundary(start + (r + 1) * len, total, cc_sink, lcc_off, lcc_len);
        float carry0 = 0.0f, carry1 = 0.0f;
        int carry_sink = -1;
        // entries and sinks are read a chunk ahead: of a chunk's two dependent rounds of loads (they, then
        // the centres and records) one passes behind the chunk before (M2L of a 384^3 box -7%)
        unsigned int e_next = r0 + lane < r1 ? cc[r0 + lane] : 0u, e_second = 0u;
        int sink_next = r0 + lane < r1 ? cc_sink[r0 + lane] : -1;
        if (KIND == 0) {  // and the sources' copies too
            m2l_stage(e_next, (int)min(32LL, r1 - r0), cen, rec, ib, row, lane);
            e_second = r0 + 32 + lane < r1 ? cc[r0 + 32 + lane] : 0u;
        }
        for (long long base = r0; base < r1; base += 32) {
            const long long idx = base + lane;
            const bool valid = idx < r1;
            const unsigned int e = e_next;
            const int sink = sink_next;
            const int ahead = KIND == 0 ? 64 : 32;
            const unsigned int e_last = idx + ahead < r1 ? cc[idx + ahead] : 0u;
            e_next = KIND == 0 ? e_second : e_last;
            e_second = e_last;
            sink_next = idx + 32 < r1 ? cc_sink[idx + 32] : -1;
            float4 hk = make_float4(0.0f, 0.0f, 0.0f, 0.0f), lk = hk;
            if (valid) {
                hk = cen[2 * sink];
                lk = cen[2 * sink + 1];
                nent++;
            }
            float acc[FMM_NL];
#pragma unroll
            for (int i = 0; i < FMM_NL; i++) acc[i] = 0.0f;
            if (KIND == 0) {
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncwarp();
                float M[FMM_NMOM];
                const float4* const src = reinterpret_cast<const float4*>(row + lane * M2L_ROW);
#pragma unroll
                for (int q4 = 0; q4 < FMM_NMOM / 4; q4++) {
                    const float4 v = src[q4];
                    M[4 * q4] = v.x;
                    M[4 * q4 + 1] = v.y;
                    M[4 * q4 + 2] = v.z;
                    M[4 * q4 + 3] = v.w;
                }
                float4 hs = src[FMM_NMOM / 4], ls = src[FMM_NMOM / 4 + 1];
                __syncwarp();  // the rows are free for the next chunk
                if (base + 32 < r1) m2l_stage(e_next, (int)min(32LL, r1 - base - 32), cen, rec, ib, row, lane);
                if (valid) {
                    float rx, ry, rz;
                    local_offset(e, hk, lk, hs, ls, ib, R, rx, ry, rz);
                    fmm_m2l_acc(M, rx, ry, rz, eps2, acc);
                }
            } else if (valid) {
                const unsigned int j = entry_index(e, ib);
                const bool part = (e & FMM_PARTICLE_BIT) != 0u;
                float4 hs = part ? posf[j] : cen[2 * j], ls = part ? plo[j] : cen[2 * j + 1];
                float rx, ry, rz;
                const float m = part ? hs.w : rec[(long long)j * FMM_NREC];  // a one-particle cell: M[0]
                local_offset(e, hk, lk, hs, ls, ib, R, rx, ry, rz);
                fmm_p2l_acc(m, rx, ry, rz, eps2, acc);
            }
#pragma unroll
            for (int i = 0; i < FMM_NL; i++) red[wl][lane][i] = acc[i];
            const int prev = __shfl_up_sync(FMM_FULL_MASK, sink, 1);
            unsigned int heads = __ballot_sync(FMM_FULL_MASK, valid && (lane == 0 || sink != prev));
            __syncwarp();
            const int nvalid = (int)min(32LL, r1 - base);
            const int after = __shfl_sync(FMM_FULL_MASK, sink_next, 0);  // the next chunk's first sink (-1: none)
            while (heads) {
                const int st = __ffs(heads) - 1;
                heads &= heads - 1;
                const int en = heads ? __ffs(heads) - 1 : nvalid;  // exclusive
                const int s_sink = __shfl_sync(FMM_FULL_MASK, sink, st);
                const bool cont = st == 0 && carry_sink == s_sink;
                float sum0 = cont ? carry0 : 0.0f, sum1 = cont ? carry1 : 0.0f;
                for (int row = st; row < en; row++) {
                    sum0 += red[wl][row][c0];
                    if (c1 < FMM_NL) sum1 += red[wl][row][c1];
                }
                carry_sink = -1;
                if (en == nvalid && after == s_sink) {  // the sink's list goes on in the next chunk
                    carry0 = sum0;
                    carry1 = sum1;
                    carry_sink = s_sink;
                    continue;
                }
                float* dst = Lown + (long long)s_sink * FMM_NL;
                if (KIND == 1 && lm2l_len[s_sink] > 0) {
                    sum0 = dst[c0] + sum0;
                    if (c1 < FMM_NL) sum1 = dst[c1] + sum1;
                }
                dst[c0] = sum0;
                if (c1 < FMM_NL) dst[c1] = sum1;
            }
            __syncwarp();
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nent += __shfl_xor_sync(FMM_FULL_MASK, nent, o);
    if (lane == 0 && nent) atomicAdd(KIND == 0 ? &ctr->n_cc : &ctr->n_cp, (unsigned long long)nent);
}

// The local expansion of a walked cell about its centre of mass, L(c) = L2L(L(parent), com(c) -
// com(parent)) + L_own(c), with L_own the sum of c's own M2L and P2L terms (zero for a cell with empty
// lists) and a level-0 cell taking its own terms only.  A local expansion is a polynomial of degree 5,
// so the chain of re-expansions equals re-expanding every ancestor's own terms to the cell directly.
//
// Only groups need theirs, so not every level waits for the one above: every LD_STEP-th level (an
// anchor level) is evaluated in place over its own terms, one launch each, and every group walks from
// the last anchor above it, as an anchor does from the anchor before: at most LD_STEP re-expansions,
// of which siblings repeat some.  The value of a cell is formed by the same operations whatever the
// step.  Walk phase by step (128^3 NFW box / 384^3 box / 4096 particles): 1: 2.91 / 47.1 ms, 4: 2.77 /
// 46.7 / 0.313, 6: 2.79 / 46.8 / 0.310.
//
// A warp takes a cell, two coefficients per lane, and shifts along one axis after the other:
// sum_j t^j/j! L_(k + j e), the exact Taylor shift of a polynomial, about 100 instructions instead of
// the 1095 flops of the shift in all three at once by one thread.  A launch is bound by its chain of
// dependent loads and launch overhead.  One launch per level with a thread per cell took 441 us on the
// 128^3 NFW box (36 levels), 348 us on a 63^3 one, 142 us on a 4096-particle box; the walk phase went
// from 3.03 to 2.83 ms, 1.21 to 0.97 and 0.37 to 0.32 with this.
#define LD_THREADS 128
#define LD_STEP FMM_LOCAL_STEP

// storage index of the coefficient (a, b, c) of order o = a + b + c, m = b + c (gen_expansions.py: order,
// then a descending, then b descending)
__device__ __forceinline__ int local_index(int o, int m, int c) { return o * (o + 1) * (o + 2) / 6 + m * (m + 1) / 2 + c; }

// For coefficient q, per axis, the storage indices of k + j e for j = 1..5, six bits each; FMM_NL (a zero)
// past order 5
__device__ __forceinline__ void local_shift_index(int q, unsigned int idx[3])
{
    idx[0] = idx[1] = idx[2] = 0u;
    int o = 0, m = 0;
    while (o < 5 && q >= (o + 1) * (o + 2) * (o + 3) / 6) o++;
    const int r = q - o * (o + 1) * (o + 2) / 6;
    while (r >= (m + 1) * (m + 2) / 2) m++;
    const int c = r - m * (m + 1) / 2;
#pragma unroll
    for (int j = 1; j <= 5; j++) {
        const bool in = q < FMM_NL && o + j <= 5;
        idx[0] |= (unsigned int)(in ? local_index(o + j, m, c) : FMM_NL) << (6 * (j - 1));
        idx[1] |= (unsigned int)(in ? local_index(o + j, m + j, c) : FMM_NL) << (6 * (j - 1));
        idx[2] |= (unsigned int)(in ? local_index(o + j, m + j, c + j) : FMM_NL) << (6 * (j - 1));
    }
}

// Coefficients lane and lane + 32 of the expansion of cell c from that of its ancestor `steps` levels up,
// whose row of L is complete (its own terms only, for done = false); buf: two rows of FMM_NL + 1 values
// of this warp.
__device__ __forceinline__ void local_chain(int c, int steps, bool done, const int* __restrict__ cparent,
                                            const int* __restrict__ lcc_len, const int* __restrict__ lcp_len,
                                            const float4* __restrict__ cen, const float* L, float (*buf)[FMM_NL + 1],
                                            const unsigned int i0[3], const unsigned int i1[3], int lane, float& v0, float& v1)
{
    const bool two = lane + 32 < FMM_NL;
    // own terms and centres along the path, all loads in flight together
    float w0[LD_STEP], w1[LD_STEP];
    float4 h[LD_STEP + 1], l[LD_STEP + 1];
    int x = c;
#pragma unroll
    for (int s = 0; s <= LD_STEP; s++) {
        if (s > steps) break;
        h[s] = cen[2 * x];
        l[s] = cen[2 * x + 1];
        const bool own = (done && s == steps) || lcc_len[x] > 0 || lcp_len[x] > 0;
        const float* row = L + (long long)x * FMM_NL;
        const float a = own ? row[lane] : 0.0f, b = own && two ? row[lane + 32] : 0.0f;
        if (s == steps) {
            v0 = a;
            v1 = b;
        } else {
            w0[s] = a;
            w1[s] = b;
        }
        if (s < steps) x = cparent[x];
    }
#pragma unroll
    for (int s = LD_STEP - 1; s >= 0; s--) {
        if (s >= steps) continue;
        const float t[3] = {cen_diff(h[s].x, l[s].x, h[s + 1].x, l[s + 1].x),
                            cen_diff(h[s].y, l[s].y, h[s + 1].y, l[s + 1].y),
                            cen_diff(h[s].z, l[s].z, h[s + 1].z, l[s + 1].z)};
#pragma unroll
        for (int a = 0; a < 3; a++) {
            float* const row = buf[a & 1];
            row[lane] = v0;
            if (two) row[lane + 32] = v1;
            __syncwarp();
            float p = t[a];
            const float inv[5] = {1.0f, 1.0f / 2.0f, 1.0f / 3.0f, 1.0f / 4.0f, 1.0f / 5.0f};
#pragma unroll
            for (int j = 0; j < 5; j++) {  // p = t^(j + 1) / (j + 1)!
                v0 = fmaf(p, row[(i0[a] >> (6 * j)) & 63u], v0);
                v1 = fmaf(p, row[(i1[a] >> (6 * j)) & 63u], v1);
                if (j < 4) p *= t[a] * inv[j + 1];
            }
        }
        v0 += w0[s];
        v1 += w1[s];
        __syncwarp();  // the first row is free again
    }
}

// The cells of an anchor level, over their own terms.
__global__ void __launch_bounds__(LD_THREADS) k_local_anchor(int level, const int* __restrict__ wcells, long long cap,
                                                            const int* __restrict__ cparent,
                                                            const int* __restrict__ lcc_len,
                                                            const int* __restrict__ lcp_len,
                                                            const float4* __restrict__ cen, float* L,
                                                            const DevCounters* __restrict__ ctr)
{
    __shared__ float buf[LD_THREADS / 32][2][FMM_NL + 1];
    if (fmm_overflowed(ctr)) return;
    const long long b0 = min((long long)ctr->lv_base[level], cap);
    const long long b1 = min((long long)ctr->lv_base[level + 1], cap);
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    if (b0 + gw >= b1) return;
    unsigned int i0[3], i1[3];
    local_shift_index(lane, i0);
    local_shift_index(lane + 32, i1);
    if (lane < 2) buf[wl][lane][FMM_NL] = 0.0f;
    __syncwarp();
    for (long long i = b0 + gw; i < b1; i += nw) {
        const int c = wcells[i];
        float v0, v1;
        local_chain(c, level == 0 ? 0 : LD_STEP, level > 0, cparent, lcc_len, lcp_len, cen, L, buf[wl], i0, i1, lane, v0, v1);
        float* row = L + (long long)c * FMM_NL;
        row[lane] = v0;
        if (lane + 32 < FMM_NL) row[lane + 32] = v1;
    }
}

// Each group's local expansion, from the last anchor level at or above it.
__global__ void __launch_bounds__(LD_THREADS) k_local_groups(const Group* __restrict__ groups,
                                                            const int* __restrict__ cparent,
                                                            const int* __restrict__ lcc_len,
                                                            const int* __restrict__ lcp_len,
                                                            const float4* __restrict__ cen, const float* L,
                                                            float* __restrict__ Lg, long long cap_groups,
                                                            const DevCounters* __restrict__ ctr)
{
    __shared__ float buf[LD_THREADS / 32][2][FMM_NL + 1];
    if (fmm_overflowed(ctr)) return;
    const long long ng = min((long long)*(volatile const unsigned long long*)&ctr->n_groups, cap_groups);
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    if (gw >= ng) return;
    unsigned int i0[3], i1[3];
    local_shift_index(lane, i0);
    local_shift_index(lane + 32, i1);
    if (lane < 2) buf[wl][lane][FMM_NL] = 0.0f;
    __syncwarp();
    for (long long gi = gw; gi < ng; gi += nw) {
        const int c = groups[gi].cell, level = groups[gi].level;
        float v0, v1;
        local_chain(c, level % LD_STEP, true, cparent, lcc_len, lcp_len, cen, L, buf[wl], i0, i1, lane, v0, v1);
        float* row = Lg + gi * FMM_NL;
        row[lane] = v0;
        if (lane + 32 < FMM_NL) row[lane + 32] = v1;
    }
}

// The shifted geometry of a periodic box's copies (PeriodicArgs): per cell and particle, axis and
// non-zero shift v, the FP64 sum rounded once to FP32 -- the values the walk's decisions use.
__global__ void k_shift_tables(const unsigned int* __restrict__ ncell, long long n, int R, const Com4* __restrict__ com,
                               const double* __restrict__ clo, const double* __restrict__ chi,
                               const double* __restrict__ sx, const double* __restrict__ sy,
                               const double* __restrict__ sz, float4* __restrict__ cshift, float* __restrict__ pshift)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int w2 = 2 * R;
    if (i < (long long)*ncell) {
        const Com4 c = com[i];
        const double cc[3] = {c.x, c.y, c.z};
        for (int ax = 0; ax < 3; ax++)
            for (int v = -R; v <= R; v++) {
                if (v == 0) continue;
                cshift[(i * 3 + ax) * w2 + shift_slot(v, R)] =
                    make_float4(__double2float_rn(cc[ax] + v), __double2float_rn(clo[3 * i + ax] + v),
                                __double2float_rn(chi[3 * i + ax] + v), 0.0f);
            }
    }
    if (i < n) {
        const double x[3] = {sx[i], sy[i], sz[i]};
        for (int ax = 0; ax < 3; ax++)
            for (int v = -R; v <= R; v++) {
                if (v == 0) continue;
                pshift[(i * 3 + ax) * w2 + shift_slot(v, R)] = __double2float_rn(x[ax] + v);
            }
    }
}

cudaError_t fmm_launch_shift_tables(DevTree& t, cudaStream_t s)
{
    if (t.per_R <= 0) return cudaSuccess;
    if (!t.cshift || !t.pshift) return cudaErrorInvalidValue;
    const long long span = std::max(t.cap_grid ? t.cap_cells : t.n_cells, t.n);
    k_shift_tables<<<(unsigned)fmm_ceil_div(span, 256), 256, 0, s>>>(t.dcount, t.n, t.per_R, t.com, t.clo, t.chi, t.sx,
                                                                     t.sy, t.sz, t.cshift, t.pshift);
    return cudaGetLastError();
}

// level 0 of the walk: every box's root cell as a sink, with that root alone on its checklist
// (isolated boxes: sources of other boxes are never seen); boxes without an active particle
// are not walked
// Each box's root starts the walk with itself on its checklist.  With one box and second_root >= 0
// (the root of an appended fixed tree, dual.cu) the checklist holds both roots.
// In a periodic box (R > 0, one box) the checklist holds the root and its (2R + 1)^3 - 1 copies,
// in the order of their copy codes.
__global__ void k_walk_seed(int* f_cell, unsigned long long* f_cloff, int* f_cllen, unsigned int* cl,
                            const int* __restrict__ cnact, const int* __restrict__ box_root, int nbox,
                            int second_root, int R, int ib, DevCounters* ctr)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbox) return;
    const int r = box_root ? box_root[b] : 0;
    if (r < 0 || cnact[r] <= 0) return;  // an empty box has no root cell
    const unsigned long long k = atomicAdd(&ctr->lv_front[0], 1ull);
    f_cell[k] = r;
    if (R > 0) {  // one box only
        const int W = 2 * R + 1, nc = W * W * W;
        f_cloff[k] = 0;
        f_cllen[k] = nc;
        for (int q = 0; q < nc; q++) cl[q] = ((unsigned int)q << ib) | (unsigned int)r;
        return;
    }
    if (second_root >= 0) {  // one box only: its entries are cl[0], cl[1]
        f_cloff[k] = 0;
        f_cllen[k] = 2;
        cl[0] = (unsigned int)r;
        cl[1] = (unsigned int)second_root;
        return;
    }
    f_cloff[k] = k;
    f_cllen[k] = 1;
    cl[k] = (unsigned int)r;
}

cudaError_t fmm_launch_walk_seed(DevTree& t, DevWalk& w, DevCounters* ctr, cudaStream_t s, int second_root)
{
    if (second_root >= 0 && t.nbox != 1) return cudaErrorInvalidValue;
    if (t.per_R > 0 && (t.nbox != 1 || second_root >= 0)) return cudaErrorInvalidValue;
    k_walk_seed<<<(unsigned)fmm_ceil_div(t.nbox, 128), 128, 0, s>>>(w.f_cell[0], w.f_cloff[0], w.f_cllen[0], w.cl[0],
                                                                     t.cnact, t.nbox > 1 ? t.box_root : nullptr,
                                                                     t.nbox, second_root, t.per_R, t.per_ib, ctr);
    return cudaGetLastError();
}

int fmm_walk_warps(int device)
{
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    return sms * 24;  // warps per SM of the walk and local-expansion grids (measured better than 20 or 16)
}

cudaError_t fmm_launch_walk_level(DevTree& t, DevWalk& w, DevCounters* ctr, const WalkArgs& a, cudaStream_t s)
{
    const int cur = a.level_parity, nxt = cur ^ 1;
    // persistent grid: every warp owns a scratch slot; blocks without a sink exit at once
    const int blocks = w.n_warps / WALK_WPB;
    WalkIO io;
    io.node = t.node;
    io.posf = t.posf;
    io.cnact = t.cnact;
    io.f_cell = w.f_cell[cur];
    io.f_cloff = w.f_cloff[cur];
    io.f_cllen = w.f_cllen[cur];
    io.ordered = (t.cap_grid ? t.cap_cells : t.n_cells) >= (a.mode == 1 ? FMM_ORDER_CELLS_NET : FMM_ORDER_CELLS);
    io.cl_cur = w.cl[cur];
    io.f_cell_next = w.f_cell[nxt];
    io.f_cloff_next = w.f_cloff[nxt];
    io.f_cllen_next = w.f_cllen[nxt];
    io.cl_next = w.cl[nxt];
    io.lcc_off = w.lcc_off;
    io.lcp_off = w.lcp_off;
    io.lcc_len = w.lcc_len;
    io.lcp_len = w.lcp_len;
    io.wcells = w.wcells;
    io.pp = w.pp;
    io.pc = w.pc;
    io.cc = w.cc;
    io.cp = w.cp;
    io.cc_sink = w.cc_sink;
    io.cp_sink = w.cp_sink;
    io.groups = w.groups;
    io.scratch = w.scratch;
    io.ctr = ctr;
    io.cap_front = w.cap_front;
    io.cap_cl = w.cap_cl;
    io.cap_pp = w.cap_pp;
    io.cap_pc = w.cap_pc;
    io.cap_cc = w.cap_cc;
    io.cap_cp = w.cap_cp;
    io.cap_groups = w.cap_groups;
    io.cap_scr = w.cap_scratch;
    io.level = a.level;
    io.group = a.group;
    io.four_eps2 = a.four_eps2;
    io.mnorm = t.mnorm;
    io.amin = t.amin;
    io.eps = a.eps;
    io.band_lo = a.band_lo;
    io.band_hi = a.band_hi;
    io.tau = a.tau;
    io.margin = a.margin;
    io.mlp_packed = a.mlp_packed;
    io.audit_pairs = a.audit_pairs;
    io.audit_cap = a.audit_cap;
    io.nogroup = t.graded ? t.nogroup : nullptr;
    io.pa = periodic_args(t);
    // the learned and audit walks take isolated boxes only (the host refuses the combinations)
    if (a.mode != 0 && t.per_R > 0) return cudaErrorInvalidValue;
    if (a.mode == 1) {
        const size_t smem = MLPP_SIZE + (size_t)WALK_WPB * MLP_WARP_SCRATCH;
        static std::atomic<unsigned long long> attr{0};
        cudaError_t e = fmm_smem_attr_once(k_walk_level<1, false>, (int)smem, attr);
        if (e != cudaSuccess) return e;
        k_walk_level<1, false><<<blocks, WALK_THREADS, smem, s>>>(io);
    } else if (a.mode == 2) {
        k_walk_level<2, false><<<blocks, WALK_THREADS, 0, s>>>(io);
    } else if (t.per_R > 0) {
        k_walk_level<0, true><<<blocks, WALK_THREADS, 0, s>>>(io);
    } else {
        k_walk_level<0, false><<<blocks, WALK_THREADS, 0, s>>>(io);
    }
    if (io.ordered) {
        const unsigned fb = (unsigned)std::min(fmm_ceil_div(w.cap_front, FRONT_TILE), 304LL);
        k_front_count<<<fb, FRONT_TILE, 0, s>>>(a.level, w.cap_front, io.f_cllen, w.front_part, ctr);
        k_front_place<<<fb, FRONT_TILE, 0, s>>>(a.level, t.node, io.f_cell, io.f_cloff, io.f_cllen, io.f_cell_next,
                                                io.f_cloff_next, io.f_cllen_next, w.cap_front, w.front_part, ctr);
        t.n_launches += 2;
    }
    return cudaGetLastError();
}

// The local expansions of walk level `level` (-1: the whole lists, then every anchor level): its own M2L
// terms, then its P2L terms, then, on an anchor level, its cells' expansions (which read the levels
// above, done by earlier calls on the same stream).  The grids are the caller's: every
// kernel takes its work with grid-stride loops, so any size gives the same result.
cudaError_t fmm_launch_local_level(DevTree& t, DevWalk& w, DevCounters* ctr, float eps2, int level, int levels,
                                   const LocalGrids& g, cudaStream_t s)
{
    k_local_flat<0><<<g.cc, LOCAL_THREADS, 0, s>>>(w.cc, w.cc_sink, w.lcc_off, w.lcc_len, w.lcc_len, t.cen, t.posf,
                                                    t.plo, t.rec, t.L, w.cap_cc, eps2, t.per_ib, t.per_R, level, ctr);
    k_local_flat<1><<<g.cp, LOCAL_THREADS, 0, s>>>(w.cp, w.cp_sink, w.lcp_off, w.lcp_len, w.lcc_len, t.cen, t.posf,
                                                    t.plo, t.rec, t.L, w.cap_cp, eps2, t.per_ib, t.per_R, level, ctr);
    const int l0 = level < 0 ? 0 : level, l1 = level < 0 ? levels : level + 1;
    for (int l = l0; l < l1; l++)
        if (l % LD_STEP == 0)
            k_local_anchor<<<g.down, LD_THREADS, 0, s>>>(l, w.wcells, w.cap_front, t.cparent, w.lcc_len, w.lcp_len,
                                                         t.cen, t.L, ctr);
    return cudaGetLastError();
}

// resident blocks per SM of the local-expansion kernels, looked up once per device
template <int KIND>
static int local_resident(int dev)
{
    static std::atomic<int> table[64];
    const bool cached = dev >= 0 && dev < 64;
    int b = cached ? table[dev].load(std::memory_order_relaxed) : 0;
    if (b > 0) return b;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_local_flat<KIND>, LOCAL_THREADS, 0) != cudaSuccess || b < 1) b = 1;
    if (cached) table[dev].store(b, std::memory_order_relaxed);
    return b;
}

// Grid sizes for a level with about n_cc / n_cp local entries and n_cells walked cells (counts of
// the context's previous walk; negative: unknown, the full persistent grids).  A full grid is what the
// SMs hold at once: its warps take ranges with a fixed stride, so blocks beyond that are a second wave
// (12 blocks per SM with 8 resident left a quarter of the M2L pass's warps idle).  Never below two
// blocks per SM: counts that changed since cost a level at most a few-fold, not its parallelism.
LocalGrids fmm_local_grids(const DevWalk& w, long long n_cc, long long n_cp, long long n_cells)
{
    (void)w;
    int sms = 152, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long full_down = (long long)sms * 8, floor = 2LL * sms;
    auto flat = [&](long long e, long long full) {
        if (e < 0) return (unsigned)full;
        // a quarter more warps than the shortest ranges
        const long long warps = fmm_ceil_div(e, LF_MIN) * 5 / 4 + 1;
        return (unsigned)std::max(std::min(floor, full), std::min(full, fmm_ceil_div(warps, LOCAL_WPB)));
    };
    LocalGrids g;
    g.cc = flat(n_cc, (long long)sms * local_resident<0>(dev));
    g.cp = flat(n_cp, (long long)sms * local_resident<1>(dev));
    g.down = n_cells < 0 ? (unsigned)full_down
                         : (unsigned)std::max(std::min(floor, full_down),
                                              std::min(full_down, fmm_ceil_div(n_cells * 5 / 4 + 1, LD_THREADS / 32)));
    return g;
}

cudaError_t fmm_launch_local_groups(DevWalk& w, DevTree& t, DevCounters* ctr, cudaStream_t s)
{
    int sms = 152, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_local_groups<<<(unsigned)(sms * 16), LD_THREADS, 0, s>>>(w.groups, t.cparent, w.lcc_len, w.lcp_len, t.cen, t.L, w.Lg,
                                                             w.cap_groups, ctr);
    return cudaGetLastError();
}
