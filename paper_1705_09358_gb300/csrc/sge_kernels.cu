// sge_kernels.cu -- sm_103a kernels of the subgraph-enumeration engine.
//
// Method (arXiv 1705.09358): RI backtracking search (Section "RI": static
// GreatestConstraintFirst order, candidates from the adjacency of the
// parent's image, pruning rules 1-4) and RI-DS (Section 4: domains D(v)
// pruned by arc consistency, forward checking of singleton domains).
//
// GPU design (not the paper's CPU work-stealing runtime):
//  * domain kernels: initialisation by one warp per 64-target bitset word or per label
//    bucket; arc consistency and forward checking iterate to their joint fixpoint in one
//    launch -- by the whole device for a few pairs, a block or a warp per pair for many --
//    or in sweeps under a host loop;
//  * split: breadth-first expansion of the search tree, up to 32 frames per
//    warp at once, to the end (its narrow part without level barriers) or until the
//    frontier holds enough frames for every resident warp;
//  * persistent search: one warp owns one depth-first search.  The CSR kernel
//    scans the candidate list (on targets with label runs the shortest run among
//    the earlier neighbours' rows) 32 candidates at a time, one per lane, spreads the
//    back-edge tests over the lanes and compacts survivors with a ballot; the bitset kernel
//    computes a whole candidate set as the AND of the parent's adjacency row,
//    the back-neighbours' rows and the filter D(mu_i), one 64-bit word per
//    lane.  Idle warps take frames from the frontier, then from a bounded
//    lock-free queue into which busy warps donate their shallowest unexplored
//    work (the paper's "steal from the back of the deque" idea without deques).
//  * every wait is bounded; cancellation, deadline and state budget are
//    checked periodically and reported through a status word.
#include "sge_internal.h"

#include <cuda/atomic>

#include <algorithm>

namespace sge {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int WARPS_PER_BLOCK = 8;
constexpr int BLOCK = WARPS_PER_BLOCK * 32;
constexpr unsigned long long CHECK_NS = 20000;         // device time between donation / abort checks
// (the timer is read every 8 iterations of the CSR kernel and every 64 of the bitset kernel,
// whose iterations are an order of magnitude cheaper)
constexpr unsigned long long CANCEL_CHECK_NS = 1000000; // device time between reads of the host cancel word
constexpr int DONATE_MIN_LEVELS = 2;     // a donated node keeps at least this many levels below it
constexpr unsigned long long IDLE_GUARD_NS = 60ull * 1000000000ull;   // 60 s idle: internal error
constexpr long long RESERVE_SPIN_LIMIT = 1 << 20;   // bounded wait for a queue cell's previous lap
constexpr int RESERVE_TICKETS = 64;                  // producer tickets tried before keeping the work
constexpr int DRAW_TRIES = 4;                        // attempts at waiting tickets before looking again later
// Idle back-off caps (ns): one warp per block polls for work at short
// intervals, the others at longer ones.  A waiting consumer polls only its own
// queue cell, so short intervals cost little and hand donated work over fast
// (measured: 256 ns / 4 us beat 1 us / 32 us by ~2.5% on the dense workload).
constexpr unsigned IDLE_BACKOFF_FAST = 256;
constexpr unsigned IDLE_BACKOFF_SLOW = 4096;

__device__ __forceinline__ uint64_t fmix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// g(u, v) of the per-match hash h(f) = fmix64(sum_u g(u, f(u))).
__device__ __forceinline__ uint64_t gterm(int u, int v) {
    return fmix64(((uint64_t)(uint32_t)u << 32 | (uint64_t)(uint32_t)v) + 0x9E3779B97F4A7C15ull);
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
    return x;
}

__device__ __forceinline__ int warp_max(int x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = max(x, __shfl_xor_sync(FULL, x, o));
    return x;
}

__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Strong (gpu-scope) loads and stores of the words warps poll and publish:
// they are ordered and always see the latest value at the point of coherence
// (L2), never a copy left in a streaming multiprocessor's L1.
__device__ __forceinline__ unsigned long long load_acquire(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_release(unsigned long long *p, unsigned long long v) {
    asm volatile("st.release.gpu.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ int load_relaxed(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// (unordered: a poll that orders nothing must not cost its SM the L1 an acquire drops)
__device__ __forceinline__ unsigned long long load_relaxed(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void set_status(int *status, int code) { atomicCAS(status, 0, code); }

// Is `c` in the sorted row of `x` (with edge label `lab` when `chk`)?
__device__ __forceinline__ bool row_has(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                                        const int32_t *__restrict__ elab, int x, int c, int lab, bool chk) {
    int lo = __ldg(rowptr + x), hi = __ldg(rowptr + x + 1);
    const int end = hi;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (__ldg(col + mid) < c) lo = mid + 1; else hi = mid;
    }
    if (lo >= end || __ldg(col + lo) != c) return false;
    return !chk || __ldg(elab + lo) == lab;
}

// Candidate source of position i (Section "RI": neighbours of M(P(mu_i));
// all of V_t, or D(mu_i) for RI-DS, when mu_i has no parent).
struct Src {
    const int32_t *ptr;   // null: candidate j is vertex j
    long long base;
    int len;
};

__device__ __forceinline__ Src cand_source(const JobDesc &J, const PosInfo &P, const int *M) {
    Src s;
    if (P.par >= 0) {
        int a = M[P.par];
        if (P.flags & POS_IN_ROW) {
            int b = __ldg(J.t.irowptr + a);
            s.ptr = J.t.icol; s.base = b; s.len = __ldg(J.t.irowptr + a + 1) - b;
        } else {
            int b = __ldg(J.t.rowptr + a);
            s.ptr = J.t.col; s.base = b; s.len = __ldg(J.t.rowptr + a + 1) - b;
        }
    } else if (J.flags & JOB_RIDS) {
        s.ptr = J.ulist; s.base = P.uoff; s.len = P.ucnt;
    } else {
        s.ptr = nullptr; s.base = 0; s.len = J.t.n;
    }
    return s;
}

// Rules 1-4 (Section "RI", pruning rules) and the RI-DS domain test for
// mapping mu_i onto candidate c.  `eidx` is c's index in the parent's row
// (for the parent-arc label), or -1.  M holds the images of positions 0..i-1.
template <bool DIR>
__device__ __forceinline__ bool feasible(const JobDesc &J, const PosInfo &P, int i, int c, long long eidx,
                                         const int *M) {
    const int2 v = __ldg(J.t.vld + c);
    if (v.x != P.lab || v.y < P.odeg) return false;                       // rules 2, 3
    if (DIR && __ldg(J.t.indeg + c) < P.ideg) return false;              // rule 3 (in)
    if (J.flags & JOB_RIDS) {                                             // v_t in D(mu_i)
        const uint64_t w = J.filt[(size_t)P.pv * J.t.dw + (c >> 6)];
        if (!((w >> (c & 63)) & 1ull)) return false;
    }
    const bool chk = (J.flags & JOB_ELAB) != 0;
    if (chk && eidx >= 0) {                                               // parent arc label
        const int l = (P.flags & POS_IN_ROW) ? __ldg(J.t.ielab + eidx) : __ldg(J.t.elab + eidx);
        if (l != P.pel) return false;
    }
    for (int b = 0; b < P.bcnt; ++b) {                                    // rule 4
        const BackEdge be = J.back[P.bbeg + b];
        const int x = M[be.pos];
        if (!DIR) {
            if (J.t.adj != nullptr && !chk) {
                const uint64_t w = __ldg(J.t.adj + (size_t)x * J.t.dw + (c >> 6));
                if (!((w >> (c & 63)) & 1ull)) return false;
            } else if (J.t.hub_slot != nullptr && !chk && __ldg(J.t.hub_slot + x) >= 0) {
                const uint64_t w = __ldg(J.t.hub_bits + (size_t)__ldg(J.t.hub_slot + x) * J.t.dw + (c >> 6));
                if (!((w >> (c & 63)) & 1ull)) return false;
            } else if (!row_has(J.t.rowptr, J.t.col, J.t.elab, x, c, be.lab_out, chk)) {
                return false;
            }
        } else {
            // arc c -> x: c is in the in-row of x; arc x -> c: c is in the out-row of x
            if ((be.dir & 1) && !row_has(J.t.irowptr, J.t.icol, J.t.ielab, x, c, be.lab_out, chk)) return false;
            if ((be.dir & 2) && !row_has(J.t.rowptr, J.t.col, J.t.elab, x, c, be.lab_in, chk)) return false;
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)                                           // rule 1 (same-label positions)
        for (uint64_t m = P.same[h]; m; m &= m - 1)
            if (M[64 * h + __ffsll((long long)m) - 1] == c) return false;
    return true;
}

__device__ __forceinline__ int find_job(const long long *off, int njobs, long long u) {
    int lo = 0, hi = njobs;  // largest j with off[j] <= u
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (off[mid] <= u) lo = mid; else hi = mid;
    }
    return lo;
}

// ------------------------------------------------- candidates of a node
//
// Position i's earlier neighbours give its constraints: number 0 is the arc to
// the parent, 1 + b back edge b (rule 4; a directed back edge names one arc).
// Each says "the candidate is in the out- or in-row of an image".  On a target
// with label runs a node's candidates are the shortest of its constraints'
// runs of lab(mu_i) -- with ties the lowest-numbered constraint's, so that every
// kernel picks the same list and a range of it means the same everywhere --
// and the other constraints are tested; without runs they are the parent's row.
// (On the 100k-vertex network a query's parent row holds 16 to 1,250 entries,
// the shortest run mostly 0 to 4.)  The node's states stay the parent's row
// length, its accepted candidates are the same set.

// One position's constants in registers.
struct PosV {
    int pv, par, lab, odeg, ideg, pel, bb, bc, flags;
};

__device__ __forceinline__ PosV load_pos(const PosInfo *p) {
    const int4 a = __ldg(reinterpret_cast<const int4 *>(p)), b = __ldg(reinterpret_cast<const int4 *>(p) + 1);
    return PosV{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, __ldg(&p->flags)};
}
static_assert(sizeof(PosInfo) == 64 && sizeof(BackEdge) == 16, "position tables are read as 16-byte words");

// A job's fields as the candidate functions read them: through its record here,
// from registers in the CSR search (CsrJob).
struct JobRef {
    const JobDesc *J;
    __device__ __forceinline__ const int32_t *rowptr() const { return J->t.rowptr; }
    __device__ __forceinline__ const int32_t *col() const { return J->t.col; }
    __device__ __forceinline__ const int32_t *elab() const { return J->t.elab; }
    __device__ __forceinline__ const int32_t *irowptr() const { return J->t.irowptr; }
    __device__ __forceinline__ const int32_t *icol() const { return J->t.icol; }
    __device__ __forceinline__ const int32_t *ielab() const { return J->t.ielab; }
    __device__ __forceinline__ const int32_t *hub_slot() const { return J->t.hub_slot; }
    __device__ __forceinline__ const uint64_t *hub_bits() const { return J->t.hub_bits; }
    __device__ __forceinline__ const uint64_t *adj() const { return J->t.adj; }
    __device__ __forceinline__ const LabelRuns *runs() const { return J->t.runs; }
    __device__ __forceinline__ const BackEdge *back() const { return J->back; }
    __device__ __forceinline__ const int32_t *ulist() const { return J->ulist; }
    __device__ __forceinline__ const int32_t *plidx() const { return J->plidx; }
    __device__ __forceinline__ int n() const { return J->t.n; }
    __device__ __forceinline__ int dw() const { return J->t.dw; }
    __device__ __forceinline__ int flags() const { return J->flags; }
};

struct Con {
    int x, in, lab;   // the candidate is in x's in-row (in != 0) or out-row, by an arc with this label
};

template <bool DIR, class V>
__device__ __forceinline__ Con constraint(const V &v, const PosV &p, int q, const int *M) {
    if (q == 0) return Con{M[p.par], DIR ? p.flags & POS_IN_ROW : 0, p.pel};
    const int4 be = __ldg(reinterpret_cast<const int4 *>(v.back() + p.bb + q - 1));
    // arc mu_i -> mu_j: the candidate is in the in-row of M_j; mu_j -> mu_i: in its out-row
    return Con{M[be.x], DIR ? be.y & 1 : 0, DIR && (be.y & 2) ? be.w : be.z};
}

struct Cand {
    const int32_t *ids;    // candidate e of the list is ids[base + e] (a run's, see li: the first of
                           // {id, degree} pair base + e); null: vertex base + e
    const int32_t *elab;   // labels beside ids (read only when edge labels are compared)
    int base, len;
    int raw;               // the node's raw candidates: the parent's row (its states)
    int skip;              // constraint the list itself satisfies, -1 for an unparented position
    int lab;               // ... and that arc's label
    int next;              // constraint with the next shortest run, -1 if there is none
    int li;                // label index of the position when the list is a run, else -1
};

// The unparented case (V_t, or D(mu_i) for RI-DS), and the parent's row on a target without runs.
template <bool DIR, class V>
__device__ __forceinline__ Cand plain_list(const V &v, const PosV &p, const PosInfo *P, const int *M) {
    Cand S;
    S.elab = nullptr;
    S.li = -1;
    S.next = -1;
    S.lab = p.pel;
    if (p.par < 0) {
        S.skip = -1;
        if (v.flags() & JOB_RIDS) {
            S.ids = v.ulist(); S.base = __ldg(&P->uoff); S.len = __ldg(&P->ucnt);
        } else {
            S.ids = nullptr; S.base = 0; S.len = v.n();
        }
    } else {
        const bool in = DIR && (p.flags & POS_IN_ROW);
        const int32_t *rp = in ? v.irowptr() : v.rowptr();
        const int a = M[p.par];
        S.skip = 0;
        S.ids = in ? v.icol() : v.col();
        S.elab = in ? v.ielab() : v.elab();
        S.base = __ldg(rp + a);
        S.len = __ldg(rp + a + 1) - S.base;
    }
    S.raw = S.len;
    return S;
}

// Start and length of constraint q's run of label index li.
template <bool DIR, class V>
__device__ __forceinline__ int run_of(const V &v, const LabelRuns *R, const PosV &p, int q, int li, const int *M,
                                      int &len) {
    const Con k = constraint<DIR>(v, p, q, M);
    const int32_t *r = (DIR && k.in ? R->irun : R->run) + (size_t)k.x * R->stride + li;
    const int b = __ldg(r);
    len = __ldg(r + 1) - b;
    return b;
}

// Candidate e of list S.
__device__ __forceinline__ int cand_id(const Cand &S, int e) {
    if (S.ids == nullptr) return S.base + e;
    return __ldg(S.ids + ((size_t)(S.base + e) << (S.li >= 0 ? 1 : 0)));
}

// First entry of ascending ids[0..n) (every other word for a run) that is at least x.
__device__ __forceinline__ int lower_bound_ids(const int32_t *ids, int n, int x, bool run = false) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(ids + ((size_t)mid << (run ? 1 : 0))) < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The parent's row of a parented position: its entries are what a checkpoint's ranges count.
template <bool DIR, class V>
__device__ __forceinline__ const int32_t *parent_row(const V &v, const PosV &p, const int *M, int &len) {
    const bool in = DIR && (p.flags & POS_IN_ROW);
    const int32_t *rp = (in ? v.irowptr() : v.rowptr()) + M[p.par];
    const int b = __ldg(rp);
    len = __ldg(rp + 1) - b;
    return (in ? v.icol() : v.col()) + b;
}

// Makes S constraint q's run.
template <bool DIR, class V>
__device__ __forceinline__ void set_run(const V &v, const LabelRuns *R, const PosV &p, const int *M, int q, int b,
                                        int len, Cand &S) {
    const Con k = constraint<DIR>(v, p, q, M);
    S.ids = reinterpret_cast<const int32_t *>(DIR && k.in ? R->icol : R->col);
    S.elab = DIR && k.in ? R->ielab : R->elab;
    S.base = b;
    S.len = len;
    S.skip = q;
    S.lab = k.lab;
}

// Entries of run S below the parent row's first: none of them is a candidate.  A range of a
// run starts at or after this one, and the part that holds it counts the node's states; so
// a later part starts later in the row too, which is how a checkpoint's row ranges tell.
template <bool DIR, class V>
__device__ __forceinline__ int run_drop(const V &v, const PosV &p, const Cand &S, const int *M) {
    int n;
    const int32_t *row = parent_row<DIR>(v, p, M, n);
    return n > 0 ? lower_bound_ids(S.ids + 2 * (size_t)S.base, S.len, __ldg(row), true) : S.len;
}

// The candidate list of position P of a node with images M[0..], found by a group of G lanes (a
// power of two; every lane of the warp calls, `sub` its lane within the group): the group's lanes
// look up the constraints' runs side by side, then agree on the shortest and the next.  With fewer
// constraints than lanes the group works as several smaller ones doing the same (most positions
// have one to three; agreeing among 32 lanes costs five rounds of shuffles, with one constraint none).
template <bool DIR, class V>
__device__ __forceinline__ Cand pick_group(const V &v, const PosV &p, const PosInfo *P, const int *M, int G, int sub) {
    Cand S = plain_list<DIR>(v, p, P, M);
    const LabelRuns *R = v.runs();
    const bool runs = R != nullptr && p.par >= 0;
    constexpr unsigned long long NONE = ~0ull;
    unsigned long long k1 = NONE, k2 = NONE;   // (length, constraint) of the shortest and next run
    int b1 = 0;
    // (the warp's groups shuffle together: as many lanes as the one with most constraints needs)
    int most = runs ? p.bc : 0;
    if (G < 32) most = (int)__reduce_max_sync(FULL, (unsigned)most);
    if (most == 0) {   // the parent's run, if any
        if (runs) {
            S.li = v.plidx()[p.pv];
            S.len = 0;
            if (S.li >= 0) {
                int len;
                const int b = run_of<DIR>(v, R, p, 0, S.li, M, len);
                set_run<DIR>(v, R, p, M, 0, b, len, S);
            }
        }
        return S;
    }
    if (most + 1 < G) G = 2 << (31 - __clz(most));
    if (runs) {
        S.li = v.plidx()[p.pv];
        if (S.li >= 0) {
#pragma unroll 4
            for (int q = sub & (G - 1); q <= p.bc; q += G) {
                int len;
                const int b = run_of<DIR>(v, R, p, q, S.li, M, len);
                const unsigned long long k = (unsigned long long)len << 32 | (unsigned)q;
                if (k < k1) { k2 = k1; k1 = k; b1 = b; }
                else if (k < k2) k2 = k;
            }
        }
    }
    for (int o = G >> 1; o >= 1; o >>= 1) {
        const unsigned long long o1 = __shfl_xor_sync(FULL, k1, o), o2 = __shfl_xor_sync(FULL, k2, o);
        const int ob = __shfl_xor_sync(FULL, b1, o);
        k2 = min(max(k1, o1), min(k2, o2));
        if (o1 < k1) { k1 = o1; b1 = ob; }
    }
    if (runs) {
        if (S.li < 0) {
            S.len = 0;
        } else {
            set_run<DIR>(v, R, p, M, (int)(unsigned)k1, b1, (int)(k1 >> 32), S);
            S.next = k2 == NONE ? -1 : (int)(unsigned)k2;
        }
    }
    return S;
}

template <bool DIR, class V>
__device__ __forceinline__ Cand pick_warp(const V &v, const PosV &p, const PosInfo *P, const int *M) {
    return pick_group<DIR>(v, p, P, M, 32, threadIdx.x & 31);
}

// The bitset row of constraint q's image, when the target keeps one and edge labels do not matter.
template <bool DIR, class V>
__device__ __forceinline__ const uint64_t *con_row(const V &v, const PosV &p, int q, const int *M) {
    if (DIR || q < 0 || (v.flags() & JOB_ELAB)) return nullptr;
    const Con k = constraint<DIR>(v, p, q, M);
    if (v.adj() != nullptr) return v.adj() + (size_t)k.x * v.dw();
    if (v.hub_slot() == nullptr) return nullptr;
    const int h = __ldg(v.hub_slot() + k.x);
    return h >= 0 ? v.hub_bits() + (size_t)h * v.dw() : nullptr;
}

// Rules 2 and 3, the domain bit and the list's own edge label for candidate c, entry e of its list.
template <bool DIR, class V>
__device__ __forceinline__ bool cand_local(const V &v, const PosV &p, const Cand &S, int c, int e) {
    if (S.li >= 0) {                                                          // rules 2 (the run's label), 3
        if (__ldg(S.ids + 2 * (size_t)(S.base + e) + 1) < p.odeg) return false;
    } else {
        const int2 r = __ldg(v.vld() + c);
        if (r.x != p.lab || r.y < p.odeg) return false;
    }
    if (DIR && __ldg(v.indeg() + c) < p.ideg) return false;                  // rule 3 (in)
    if (v.flags() & JOB_RIDS) {                                               // v_t in D(mu_i)
        const uint64_t w = v.filt()[(size_t)p.pv * v.dw() + (c >> 6)];
        if (!((w >> (c & 63)) & 1ull)) return false;
    }
    return !(v.flags() & JOB_ELAB) || S.skip < 0 || __ldg(S.elab + S.base + e) == S.lab;
}

// Is candidate c where constraint q wants it (rule 4)?
template <bool DIR, class V>
__device__ __forceinline__ bool con_holds(const V &v, const PosV &p, int q, int li, int c, const int *M) {
    const Con k = constraint<DIR>(v, p, q, M);
    const bool chk = (v.flags() & JOB_ELAB) != 0;
    if (!DIR && !chk) {
        if (v.adj() != nullptr) return (__ldg(v.adj() + (size_t)k.x * v.dw() + (c >> 6)) >> (c & 63)) & 1ull;
        if (v.hub_slot() != nullptr) {
            const int h = __ldg(v.hub_slot() + k.x);
            if (h >= 0) return (__ldg(v.hub_bits() + (size_t)h * v.dw() + (c >> 6)) >> (c & 63)) & 1ull;
        }
    }
    // binary search in x's run of the position's label, else in its whole row
    const LabelRuns *R = v.runs();
    const bool in = DIR && k.in, run = R != nullptr && li >= 0;
    const int32_t *at = run ? (in ? R->irun : R->run) + (size_t)k.x * R->stride + li
                            : (in ? v.irowptr() : v.rowptr()) + k.x;
    const int32_t *col = run ? reinterpret_cast<const int32_t *>(in ? R->icol : R->col) : (in ? v.icol() : v.col());
    const int step = run ? 1 : 0;   // (a run's ids are every other word)
    int lo = __ldg(at), hi = __ldg(at + 1);
    const int end = hi;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(col + ((size_t)mid << step)) < c) lo = mid + 1; else hi = mid;
    }
    if (lo >= end || __ldg(col + ((size_t)lo << step)) != c) return false;
    return !chk || __ldg((run ? (in ? R->ielab : R->elab) : (in ? v.ielab() : v.elab())) + lo) == k.lab;
}

// Rule 1 against the positions named in `same`.
__device__ __forceinline__ bool unused(const PosInfo *P, int c, const int *M) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
        for (uint64_t m = __ldg(&P->same[h]); m; m &= m - 1)
            if (M[64 * h + __ffsll((long long)m) - 1] == c) return false;
    return true;
}

// Up to this many (candidate, constraint) tests of a chunk are spread over the warp's lanes: four
// rounds of them (64, 256 and 1,024 measured alike on deep, network, directed and molecule batches).
constexpr int SPREAD_TESTS = 128;

// Warp-collective: the candidates of entries [x0, x0 + 32) below `end` of list S that pass all
// rules, as a ballot; `c` receives this lane's candidate (-1 beyond the list).  Each lane makes
// its candidate's local tests; the few that remain are tested against the constraints with the
// lanes spread over (candidate, constraint) pairs, so that a node costs a handful of dependent
// loads however many earlier neighbours it has; a chunk with many left tests them lane by lane,
// leaving at the first that fails.  Cs: 32 ints of shared memory of this warp.
template <bool DIR, class V>
__device__ __forceinline__ unsigned cand_chunk(const V &v, const PosV &p, const PosInfo *P, const Cand &S, int x0,
                                               int end, const int *M, int *Cs, int &c) {
    const int lane = threadIdx.x & 31;
    const int e = x0 + lane;
    bool ok = false;
    c = -1;
    if (e < end) {
        c = cand_id(S, e);
        ok = cand_local<DIR>(v, p, S, c, e);
    }
    const unsigned loc = __ballot_sync(FULL, ok);
    const int nq = p.par >= 0 ? p.bc : 0;   // constraints left to test (the list satisfies one)
    if (loc && nq) {
        const int left = __popc(loc);
        if (left * nq <= SPREAD_TESTS) {
            const int r = __popc(loc & ((1u << lane) - 1u));
            if (ok) Cs[r] = c;
            __syncwarp();
            unsigned bad = 0;
            for (int t = lane; t < left * nq; t += 32) {
                const int q = t / left, x = t - q * left;
                if (!con_holds<DIR>(v, p, q + (q >= S.skip ? 1 : 0), S.li, Cs[x], M)) bad |= 1u << x;
            }
            bad = __reduce_or_sync(FULL, bad);
            if (ok) ok = !((bad >> r) & 1u);
        } else if (ok) {
            for (int q = 0; ok && q <= p.bc; ++q) ok = q == S.skip || con_holds<DIR>(v, p, q, S.li, c, M);
        }
    }
    if (ok) ok = unused(P, c, M);
    return __ballot_sync(FULL, ok);
}

// A frame's range [beg, end) (beg < 0: everything) as entries [lo, hi) of list S: as it stands
// (clipped) unless S is a run and the range counts in the parent's row -- both ascend, so the
// row range is an interval of ids.  Returns whether this part counts the node's states.
template <bool DIR, class V>
__device__ __forceinline__ bool list_range(const V &v, const PosV &p, const Cand &S, const int *M, int beg, int end,
                                           bool in_run, int &lo, int &hi) {
    lo = beg >= 0 ? beg : 0;
    hi = beg >= 0 ? min(end, S.len) : S.len;   // (S is never longer than the parent's row)
    if (beg < 0) return true;
    if (in_run) {
        if (S.li < 0) {   // the label is absent: no entry
            lo = hi = 0;
            return beg == 0;
        }
        const int drop = run_drop<DIR>(v, p, S, M);
        lo = max(beg, drop);
        return beg <= drop && drop < end;
    }
    if (S.li < 0 || (beg == 0 && end >= S.raw)) return beg == 0;
    int len;
    const int32_t *row = parent_row<DIR>(v, p, M, len);
    const int e = min(end, len);
    if (beg >= e) {
        lo = hi = 0;
    } else {
        lo = lower_bound_ids(S.ids + 2 * (size_t)S.base, S.len, __ldg(row + beg), true);
        hi = lower_bound_ids(S.ids + 2 * (size_t)S.base, S.len, __ldg(row + e - 1) + 1, true);
    }
    return beg == 0;
}

// The other way: entries [lo, hi) of list S (lo < hi) as a range of the parent's row.
template <bool DIR, class V>
__device__ __forceinline__ void row_range(const V &v, const PosV &p, const Cand &S, const int *M, int lo, int hi,
                                          int &beg, int &end) {
    beg = lo;
    end = hi;
    if (S.li < 0) return;
    int len;
    const int32_t *row = parent_row<DIR>(v, p, M, len);
    // (an entry of another constraint's run need not be in the parent's row: bounds by id)
    beg = lower_bound_ids(row, len, cand_id(S, lo));
    end = lower_bound_ids(row, len, cand_id(S, hi - 1) + 1);
}

// Write one match row (images of pattern vertices 0..k-1) for enumeration.
__device__ __forceinline__ void emit_match(const JobDesc &J, const int *M, int last_pos, int c) {
    if ((long long)load_relaxed(J.mlen) >= J.mcap) return;   // (full: the counters tell how many there are)
    unsigned long long slot = atomicAdd(J.mlen, 1ull);
    if ((long long)slot >= J.mcap) return;
    int32_t *row = J.mbuf + (size_t)slot * J.k;
    for (int t = 0; t < last_pos; ++t) row[J.pos[t].pv] = M[t];
    row[J.pos[last_pos].pv] = c;
}

// ================================================================ domains

// Each pattern vertex's label index among its job's target labels (-1: absent),
// for the jobs that keep one: one block per job, one thread per vertex.
__global__ void __launch_bounds__(KMAX) k_label_index(const JobDesc *jobs) {
    const JobDesc &J = jobs[blockIdx.x];
    const int u = threadIdx.x;
    if (J.plidx == nullptr || u >= J.p.k) return;
    const int lab = J.p.lab[u];
    int lo = 0, hi = J.t.nlab;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(J.t.labs + mid) < lab) lo = mid + 1; else hi = mid;
    }
    const_cast<int32_t *>(J.plidx)[u] = lo < J.t.nlab && __ldg(J.t.labs + lo) == lab ? lo : -1;
}

// Initial domain of pattern vertex v on a target with label buckets: the prefix of
// lab(v)'s bucket with degree at least v's (descending order), then, for RI-DS, the
// label-degree support test of k_domain_init; bits set with atomicOr into the zeroed filter.
// BUCKET_PARTS warps share a prefix (a frequent label's holds a quarter of the target, and one
// warp walking it through the dependent table look-ups set the launch's length).
constexpr int BUCKET_PARTS = 16;
__global__ void __launch_bounds__(BLOCK) k_domain_init_buckets(const JobDesc *jobs, const long long *vert_off,
                                                               int njobs, long long nverts) {
    const long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (g >= nverts) return;
    const int j = find_job(vert_off, njobs, g);
    const JobDesc &J = jobs[j];
    if (J.filt == nullptr || J.t.lbuck == nullptr) return;
    const int v = (int)(g - vert_off[j]);
    const int lab = J.p.lab[v], od = J.p.odeg[v];
    int lo = 0, hi = J.t.nlab;   // lab(v)'s bucket
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(J.t.labs + mid) < lab) lo = mid + 1; else hi = mid;
    }
    if (lo >= J.t.nlab || __ldg(J.t.labs + lo) != lab) return;   // label absent: empty domain
    const int b0 = __ldg(J.t.lbstart + lo), b1 = __ldg(J.t.lbstart + lo + 1);
    int e = b0, f = b1;          // first bucket position with degree below od (degrees descend)
    while (e < f) {
        const int mid = (e + f) >> 1;
        if (__ldg(J.t.lbdeg + mid) >= od) e = mid + 1; else f = mid;
    }
    const bool nbcheck = (J.flags & JOB_RIDS) && !(J.flags & JOB_ELAB) && J.t.nbmax != nullptr && J.plidx != nullptr;
    uint64_t *Fv = J.filt + (size_t)v * J.t.dw;
    for (int x = b0 + blockIdx.y * 32 + lane; x < e; x += 32 * BUCKET_PARTS) {
        const int t = __ldg(J.t.lbuck + x);
        bool ok = true;
        if (nbcheck) {
            for (int pe = J.p.rowptr[v]; pe < J.p.rowptr[v + 1] && ok; ++pe) {
                const int pu = J.p.col[pe];
                const int li = J.plidx[pu];
                ok = li >= 0 && __ldg(J.t.nbmax + (size_t)li * J.t.n + t) >= J.p.odeg[pu];
            }
        }
        if (ok) atomicOr((unsigned long long *)(Fv + (t >> 6)), 1ull << (t & 63));
    }
}

// D(v) initialisation (Section 4): equal label, in/out-degree at least v's.
// For RI it is exactly the rule 2-3 filter.  One warp per 32 consecutive 64-bit words.
constexpr int INIT_WORDS_PER_WARP = 32;   // most consecutive filter words one warp of k_domain_init writes
static_assert(INIT_WORDS_PER_WARP <= 32, "k_domain_init copies a warp's words one per lane");

__global__ void __launch_bounds__(BLOCK) k_domain_init(const JobDesc *jobs, const long long *unit_off, int njobs,
                                                       long long nunits, int wpw) {
    const long long u0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * wpw;
    const int lane = threadIdx.x & 31;
    if (u0 >= nunits) return;
    // the warp's words are consecutive units: find the job once, then step over its
    // boundaries; (v, q) = (pattern vertex, word) steps along with u (a job holds
    // k x dw < 2^15 units, so 32-bit arithmetic).  The job's fields are read once per job
    // and the vertex's once per vertex, not once per word.
    int j = find_job(unit_off, njobs, u0);
    {
        // when every word of the warp's range is a copy of a label-degree mask row (see
        // below), the lanes copy one word each at once instead of the warp stepping word by word
        const long long u = u0 + lane;
        bool copyable = true;
        uint64_t *dst = nullptr;
        uint64_t word = 0;
        if (u < nunits && u < u0 + wpw) {
            int jl = j;
            while (jl + 1 < njobs && unit_off[jl + 1] <= u) ++jl;
            const JobDesc &J = jobs[jl];
            if (J.filt != nullptr && J.t.lbuck == nullptr) {
                const bool nbc = (J.flags & JOB_RIDS) && !(J.flags & JOB_ELAB) && J.t.nbmax != nullptr &&
                                 J.plidx != nullptr;
                const int dwl = J.t.dw, local = (int)(u - unit_off[jl]);
                const int vl = local / dwl, ql = local - vl * dwl;
                const int odl = J.p.odeg[vl];
                if (nbc || (J.flags & JOB_DIRECTED) || J.t.ldm == nullptr || odl >= LDM_DEGREES) {
                    copyable = false;
                } else {
                    const int labl = J.p.lab[vl];
                    int lo = 0, hi = J.t.nlab;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (__ldg(J.t.labs + mid) < labl) lo = mid + 1; else hi = mid;
                    }
                    if (lo < J.t.nlab && __ldg(J.t.labs + lo) == labl)
                        word = __ldg(J.t.ldm + ((size_t)lo * LDM_DEGREES + odl) * dwl + ql);
                    dst = J.filt + (size_t)vl * dwl + ql;
                }
            }
        }
        if (__all_sync(FULL, copyable)) {
            if (dst != nullptr) *dst = word;
            return;
        }
    }
    int jcur = -1, v = -1, q = 0, vcur = -1;
    bool skip = true, DIR = false, nbcheck = false;
    int dw = 1, n = 0, lab = 0, od = 0, id = 0;
    const int2 *vld = nullptr;
    const int32_t *indeg = nullptr;
    uint64_t *filt = nullptr;
    // without the neighbour test, D(v) initialised = the target's label-degree mask row of
    // (lab(v), deg(v)) when it has one: a copy (mrow null and mempty: lab(v) absent)
    const uint64_t *mrow = nullptr;
    bool mempty = false;
    for (long long u = u0; u < u0 + wpw && u < nunits; ++u) {
        while (j + 1 < njobs && unit_off[j + 1] <= u) ++j;
        const JobDesc &J = jobs[j];
        if (j != jcur) {
            jcur = j;
            skip = J.filt == nullptr || J.t.lbuck != nullptr;   // (bucket targets: k_domain_init_buckets)
            DIR = (J.flags & JOB_DIRECTED) != 0;
            // RI-DS on an undirected target without edge labels: a candidate t also needs, for
            // every pattern neighbour u of v, a neighbour of its own with u's label and at least
            // u's degree.  That is arc consistency's test against the domains as initialised, so
            // dropping the failures here removes only candidates the first sweep would remove;
            // their rows, which the sweep would scan to the end, are never read.
            nbcheck = (J.flags & JOB_RIDS) && !(J.flags & JOB_ELAB) && !DIR && J.t.nbmax != nullptr &&
                      J.plidx != nullptr;
            dw = J.t.dw;
            n = J.t.n;
            vld = J.t.vld;
            indeg = J.t.indeg;
            filt = J.filt;
            const int local = (int)(u - unit_off[j]);
            v = local / dw;
            q = local - v * dw;
            vcur = -1;
        } else if (++q == dw) {
            q = 0;
            ++v;
        }
        if (skip) continue;
        if (v != vcur) {
            vcur = v;
            lab = J.p.lab[v];
            od = J.p.odeg[v];
            id = DIR ? J.p.ideg[v] : 0;
            mrow = nullptr;
            mempty = false;
            if (!nbcheck && !DIR && J.t.ldm != nullptr && od < LDM_DEGREES) {
                int lo = 0, hi = J.t.nlab;   // lab(v)'s index among the target's labels
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (__ldg(J.t.labs + mid) < lab) lo = mid + 1; else hi = mid;
                }
                if (lo < J.t.nlab && __ldg(J.t.labs + lo) == lab)
                    mrow = J.t.ldm + ((size_t)lo * LDM_DEGREES + od) * dw;
                else
                    mempty = true;
            }
        }
        if (mrow != nullptr || mempty) {
            if (lane == 0) filt[(size_t)v * dw + q] = mempty ? 0ull : __ldg(mrow + q);
            continue;
        }
        unsigned long long word = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = q * 64 + h * 32 + lane;
            bool ok = false;
            if (t < n) {
                const int2 x = __ldg(vld + t);
                ok = x.x == lab && x.y >= od && (!DIR || __ldg(indeg + t) >= id);
            }
            if (nbcheck && __any_sync(FULL, ok)) {
                for (int e = J.p.rowptr[v]; e < J.p.rowptr[v + 1]; ++e) {
                    const int pu = J.p.col[e];
                    const int li = J.plidx[pu];   // lab(pu)'s index among the target's labels, -1 if absent
                    if (ok) ok = li >= 0 && __ldg(J.t.nbmax + (size_t)li * n + t) >= J.p.odeg[pu];
                }
            }
            word |= (unsigned long long)__ballot_sync(FULL, ok) << (32 * h);
        }
        if (lane == 0) filt[(size_t)v * dw + q] = word;
    }
}

// Where a target vertex t may find support for a pattern edge into vertex u: its row (out- or
// in-), or, on a target with label runs, the run of u's label in it.
struct AcList {
    const int32_t *ids;   // entry f is ids[f << shift]
    const int32_t *lab;   // edge labels, one per entry
    int len, shift;
};

__device__ __forceinline__ AcList ac_list(const JobDesc &J, int u, int t, bool in) {
    AcList A;
    const LabelRuns *R = J.t.runs;
    if (R != nullptr && J.plidx != nullptr) {
        const int li = J.plidx[u];
        A.ids = nullptr; A.lab = nullptr; A.len = 0; A.shift = 1;
        if (li < 0) return A;   // no vertex carries u's label
        const int32_t *r = (in ? R->irun : R->run) + (size_t)t * R->stride + li;
        const int b = __ldg(r);
        A.len = __ldg(r + 1) - b;
        A.ids = reinterpret_cast<const int32_t *>((in ? R->icol : R->col) + b);
        A.lab = (in ? R->ielab : R->elab) + b;
    } else {
        const int32_t *rp = (in ? J.t.irowptr : J.t.rowptr) + t;
        const int b = __ldg(rp);
        A.len = __ldg(rp + 1) - b;
        A.ids = (in ? J.t.icol : J.t.col) + b;
        A.lab = (in ? J.t.ielab : J.t.elab) + b;
        A.shift = 0;
    }
    return A;
}

// Is one of the first n entries of A (with edge label bl when `chk`) in the domain Du?  Four entries'
// ids, then their domain words, are in flight together: the scan is a chain of such pairs of loads.
__device__ __forceinline__ bool ac_scan(const AcList &A, int n, const uint64_t *Du, bool chk, int bl) {
    for (int f0 = 0; f0 < n; f0 += 4) {
        int y[4];
        uint64_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = f0 + i < n ? __ldg(A.ids + ((size_t)(f0 + i) << A.shift)) : -1;
        if (chk) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (y[i] >= 0 && __ldg(A.lab + f0 + i) != bl) y[i] = -1;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = y[i] >= 0 ? Du[y[i] >> 6] : 0ull;
        bool any = false;
#pragma unroll
        for (int i = 0; i < 4; ++i) any = any || ((w[i] >> (y[i] & 63)) & 1ull);
        if (any) return true;
    }
    return false;
}

// Arc consistency of one candidate (Section 4): does target vertex t keep, for every pattern
// edge at v, a compatible target edge into the other endpoint's domain?
__device__ __forceinline__ bool ac_supported(const JobDesc &J, int v, int t, bool DIR, bool chk) {
    const int dw = J.t.dw;
    for (int pass = 0; pass < (DIR ? 2 : 1); ++pass) {
        const int32_t *prow = pass ? J.p.irowptr : J.p.rowptr;
        const int32_t *pcol = pass ? J.p.icol : J.p.col;
        const int32_t *pel = pass ? J.p.ielab : J.p.elab;
        for (int e = prow[v], ee = prow[v + 1]; e < ee; ++e) {
            const int u = pcol[e];
            const AcList A = ac_list(J, u, t, pass != 0);
            if (!ac_scan(A, A.len, J.filt + (size_t)u * dw, chk, chk ? pel[e] : 0)) return false;
        }
    }
    return true;
}

// A list longer than AC_WARP_LIST is searched by the whole warp (ac_supported_warp) -- unless the
// domains at the other ends of v's pattern edges are dense (each at least 1/AC_DENSE of the
// target), where a scan finds support within a few entries: then the candidate's own lane scans
// AC_LANE_SCAN entries first.  Lists longer than AC_WARP_DIRECT always go to the warp.
constexpr int AC_WARP_LIST = 48;
constexpr int AC_LANE_SCAN = 32;
constexpr int AC_WARP_DIRECT = 512;

// Warp-collective: are the pattern edges at v with long lists supported at t?  For each the 32
// lanes stride the list and a ballot says whether any of them found support.
__device__ __forceinline__ bool ac_supported_warp(const JobDesc &J, int v, int t, bool DIR, bool chk) {
    const int lane = threadIdx.x & 31;
    const int dw = J.t.dw;
    for (int pass = 0; pass < (DIR ? 2 : 1); ++pass) {
        const int32_t *prow = pass ? J.p.irowptr : J.p.rowptr;
        const int32_t *pcol = pass ? J.p.icol : J.p.col;
        const int32_t *pel = pass ? J.p.ielab : J.p.elab;
        for (int e = prow[v], ee = prow[v + 1]; e < ee; ++e) {
            const int u = pcol[e], bl = chk ? pel[e] : 0;
            const AcList A = ac_list(J, u, t, pass != 0);
            if (A.len <= AC_WARP_LIST) continue;   // (the candidate's lane has found its support)
            const uint64_t *Du = J.filt + (size_t)u * dw;
            bool found = false;
            for (int f0 = 0; f0 < A.len && !found; f0 += 64) {
                bool ok = false;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int f = f0 + 32 * i + lane;
                    if (f < A.len) {
                        const int y = __ldg(A.ids + ((size_t)f << A.shift));
                        ok = ok || ((!chk || __ldg(A.lab + f) == bl) && ((Du[y >> 6] >> (y & 63)) & 1ull));
                    }
                }
                found = __any_sync(FULL, ok);
            }
            if (!found) return false;
        }
    }
    return true;
}

// Lane-local part of the arc-consistency test of candidate t of D(v): whether to drop it, or
// (`heavy`) to have the warp look at its long lists.
__device__ __forceinline__ bool ac_lane_check(const JobDesc &J, int v, int t, bool DIR, bool chk, bool dense,
                                              bool &heavy) {
    const int dw = J.t.dw;
    heavy = false;
    for (int pass = 0; pass < (DIR ? 2 : 1); ++pass) {
        const int32_t *prow = pass ? J.p.irowptr : J.p.rowptr;
        const int32_t *pcol = pass ? J.p.icol : J.p.col;
        const int32_t *pel = pass ? J.p.ielab : J.p.elab;
        for (int e = prow[v], ee = prow[v + 1]; e < ee; ++e) {
            const int u = pcol[e];
            const AcList A = ac_list(J, u, t, pass != 0);
            const bool all = A.len <= AC_WARP_LIST;
            const int n = all ? A.len : dense && A.len <= AC_WARP_DIRECT ? AC_LANE_SCAN : 0;
            if (ac_scan(A, n, J.filt + (size_t)u * dw, chk, chk ? pel[e] : 0)) continue;
            if (all) {
                heavy = false;
                return true;
            }
            heavy = true;
        }
    }
    return false;
}

// The same sweep over explicit candidate lists: one lane per listed candidate of
// the listed entries {job, pattern vertex, global vertex, list start}; a removed
// candidate is cleared from D(v) and its list slot.  A lane tests a candidate with
// a short row itself; the warp then takes its lanes' long-row candidates one at a
// time together, so a hub's row is read 32 entries per step instead of one.
__global__ void __launch_bounds__(BLOCK, 1) k_domain_ac_cand(const JobDesc *jobs, const int4 *ent, const long long *eoff,
                                                          int nent, long long ncand, int32_t *cand, int *changed,
                                                          unsigned char *vchanged) {
    const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if ((x & ~31ll) >= ncand) return;   // warp-uniform: a warp with any candidate stays whole
    const int lane = threadIdx.x & 31;
    int jidx = 0, v = 0, g = 0, t = -1;
    bool dense_v = false;
    int32_t *slot = nullptr;
    if (x < ncand) {
        const int i = find_job(eoff, nent, x);
        const int4 E = ent[i];
        jidx = E.x; v = E.y & (AC_ENT_DENSE - 1); g = E.z;
        dense_v = (E.y & AC_ENT_DENSE) != 0;
        slot = cand + (long long)E.w + (x - eoff[i]);
        t = *slot;
    }
    bool drop = false, heavy = false;
    if (t >= 0) {
        const JobDesc &J = jobs[jidx];
        uint64_t *wp = J.filt + (size_t)v * J.t.dw + (t >> 6);
        if (!(*wp & (1ull << (t & 63)))) {
            *slot = -1;                                  // removed by forward checking
        } else {
            drop = ac_lane_check(J, v, t, (J.flags & JOB_DIRECTED) != 0, (J.flags & JOB_ELAB) != 0, dense_v, heavy);
        }
    }
    unsigned hv = __ballot_sync(FULL, heavy);
    while (hv) {
        const int L = __ffs(hv) - 1;
        hv &= hv - 1;
        const int jl = __shfl_sync(FULL, jidx, L), vl = __shfl_sync(FULL, v, L), tl = __shfl_sync(FULL, t, L);
        const JobDesc &J = jobs[jl];
        const bool sup = ac_supported_warp(J, vl, tl, (J.flags & JOB_DIRECTED) != 0, (J.flags & JOB_ELAB) != 0);
        if (lane == L) drop = !sup;
    }
    if (drop) {                                          // unsupported: remove t from D(v)
        const JobDesc &J = jobs[jidx];
        atomicAnd((unsigned long long *)(J.filt + (size_t)v * J.t.dw + (t >> 6)), ~(1ull << (t & 63)));
        *slot = -1;
        *changed = 1;
        vchanged[g] = 1;
    }
}

// One arc-consistency sweep (Section 4): drop t from D(v) when a pattern
// edge at v has no compatible target edge at t into the other endpoint's
// domain.  Removals are applied in place (monotone), so sweeping until no
// word changes reaches the unique greatest fixpoint.  A sweep visits only
// the listed (job, pattern vertex) entries -- those with a neighbour whose
// domain shrank in the previous sweep -- one warp per 64-target word, and
// marks every domain it shrinks in vchanged.
__global__ void __launch_bounds__(BLOCK, 1) k_domain_ac(const JobDesc *jobs, const int4 *ent, const long long *eoff,
                                                     int nent, long long nunits, int *changed,
                                                     unsigned char *vchanged) {
    const long long u = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (u >= nunits) return;
    const int i = find_job(eoff, nent, u);
    const int4 E = ent[i];   // {job, pattern vertex, global vertex index, 0}
    const JobDesc &J = jobs[E.x];
    if (J.filt == nullptr || !(J.flags & JOB_RIDS)) return;
    const bool DIR = (J.flags & JOB_DIRECTED) != 0;
    const int v = E.y & (AC_ENT_DENSE - 1), q = (int)(u - eoff[i]);
    uint64_t *wp = J.filt + (size_t)v * J.t.dw + q;
    const uint64_t word = *wp;
    if (word == 0) return;
    const bool chk = (J.flags & JOB_ELAB) != 0;
    const int dw = J.t.dw;
    unsigned long long keep = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int bit = h * 32 + lane;
        const int t = q * 64 + bit;
        bool ok = (word >> bit) & 1ull;
        if (ok) {
            for (int e = J.p.rowptr[v]; ok && e < J.p.rowptr[v + 1]; ++e) {
                const int uu = J.p.col[e], bl = chk ? J.p.elab[e] : 0;
                const uint64_t *Du = J.filt + (size_t)uu * dw;
                bool found = false;
                for (int f = __ldg(J.t.rowptr + t), fe = __ldg(J.t.rowptr + t + 1); f < fe; ++f) {
                    const int y = __ldg(J.t.col + f);
                    if ((!chk || __ldg(J.t.elab + f) == bl) && ((Du[y >> 6] >> (y & 63)) & 1ull)) { found = true; break; }
                }
                ok = found;
            }
            if (DIR) {
                for (int e = J.p.irowptr[v]; ok && e < J.p.irowptr[v + 1]; ++e) {
                    const int uu = J.p.icol[e], bl = chk ? J.p.ielab[e] : 0;
                    const uint64_t *Du = J.filt + (size_t)uu * dw;
                    bool found = false;
                    for (int f = __ldg(J.t.irowptr + t), fe = __ldg(J.t.irowptr + t + 1); f < fe; ++f) {
                        const int y = __ldg(J.t.icol + f);
                        if ((!chk || __ldg(J.t.ielab + f) == bl) && ((Du[y >> 6] >> (y & 63)) & 1ull)) { found = true; break; }
                    }
                    ok = found;
                }
            }
        }
        keep |= (unsigned long long)__ballot_sync(FULL, ok) << (32 * h);
    }
    if (lane == 0 && keep != word) {
        atomicAnd((unsigned long long *)wp, keep);
        *changed = 1;
        vchanged[E.z] = 1;
    }
}

// Forward checking (Section 4.2): the target node of a singleton domain is
// removed from every other domain, repeated until no new singleton appears.
// One block per job, starting from the domain sizes: each round takes the
// singletons not yet propagated, finds each one's element (one warp scans
// its words), and clears that element's word in every other domain,
// counting the sizes down (all singletons of a round propagate together).
__global__ void __launch_bounds__(BLOCK) k_domain_fc(const JobDesc *jobs, const long long *vert_off,
                                                     const long long *sizes, int *changed, unsigned char *vchanged) {
    __shared__ int size[KMAX];
    __shared__ int elem[KMAX];
    __shared__ unsigned char done[KMAX];
    __shared__ int newu[KMAX];
    __shared__ int nnew;
    const JobDesc &J = jobs[blockIdx.x];
    if (J.filt == nullptr || !(J.flags & JOB_FC)) return;
    const int k = J.k, dw = J.t.dw;
    const long long vo = vert_off[blockIdx.x];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int v = threadIdx.x; v < k; v += blockDim.x) {
        size[v] = (int)sizes[vo + v];   // exact, counted down on every removal
        done[v] = 0;
    }
    __syncthreads();
    for (int round = 0; round <= k; ++round) {
        if (threadIdx.x == 0) nnew = 0;
        __syncthreads();
        for (int v = threadIdx.x; v < k; v += blockDim.x)
            if (size[v] == 1 && !done[v]) {
                done[v] = 1;
                newu[atomicAdd(&nnew, 1)] = v;
            }
        __syncthreads();
        const int nn = nnew;
        if (nn == 0) break;
        for (int s = wid; s < nn; s += nwarps) {
            const int u = newu[s];
            int found = -1;
            for (int q0 = 0; q0 < dw && found < 0; q0 += 32) {
                const int q = q0 + lane;
                const uint64_t w = q < dw ? J.filt[(size_t)u * dw + q] : 0ull;
                const unsigned b = __ballot_sync(FULL, w != 0);
                if (b) {
                    const int L = __ffs(b) - 1;
                    const uint64_t wl = __shfl_sync(FULL, w, L);
                    found = (q0 + L) * 64 + __ffsll((long long)wl) - 1;
                }
            }
            if (lane == 0) elem[u] = found;
        }
        __syncthreads();
        for (int x = threadIdx.x; x < nn * k; x += blockDim.x) {
            const int u = newu[x / k], v = x % k, t = elem[u];
            if (v == u || t < 0) continue;
            unsigned long long *wp = reinterpret_cast<unsigned long long *>(J.filt + (size_t)v * dw + (t >> 6));
            const unsigned long long bit = 1ull << (t & 63);
            if (atomicAnd(wp, ~bit) & bit) {
                atomicSub(&size[v], 1);
                vchanged[vo + v] = 1;
                *changed = 1;
            }
        }
        __syncthreads();
    }
}

// Arc consistency alternating with forward checking to their joint fixpoint
// (Section 4, Section 4.2), all of one job inside one block: no host round
// trip between sweeps, so a batch of many small jobs costs one launch.  A
// sweep re-checks D(v) only for the vertices whose pattern neighbours' domains
// shrank in the previous sweep (all vertices first); when arc consistency
// holds, one forward-checking round clears the element of every new singleton
// from the other domains, and the loop goes on until neither changes anything.
// Removals are monotone deletions, so this schedule reaches the same unique
// greatest fixpoint as any other.  A forward-checking round that finds an
// empty domain ends the job (it has no match).  Blocks take jobs from a counter.
// A sweep visits a dirty vertex's candidates either word by word (small
// targets: `cand` null) or through its candidate list (large targets, whose
// domain words are mostly empty: slots [cstart[g], cstart[g] + csize[g]) of
// `cand`, g = vert_off[job] + v, a removed candidate's slot set to -1), 32
// slots per warp step so that a candidate with a long row is checked by the
// whole warp.
constexpr int FIXPOINT_BIG_BLOCK = 1024;   // threads per block of k_domain_fixpoint when pairs are few
constexpr int FIXPOINT_SMALL_BLOCK = 128;  // ... and when they are many
constexpr int FP_CHUNK = 1024;             // domain words scanned at once by k_domain_fixpoint
static_assert(FP_CHUNK % FIXPOINT_BIG_BLOCK == 0 && FP_CHUNK % FIXPOINT_SMALL_BLOCK == 0,
              "a fixpoint block scans FP_CHUNK words in whole rounds of one word per thread");

// Exclusive scan of one int per thread over the block (up to 1024 threads);
// `total` receives the block's sum.  wsum: 32 ints of shared memory.
__device__ __forceinline__ int block_scan_int(int x, int *wsum, int &total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int s = lane < nw ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nw) wsum[lane] = s;
    }
    __syncthreads();
    total = wsum[nw - 1];
    const int before = wid ? wsum[wid - 1] : 0;
    __syncthreads();   // wsum may be reused at once
    return before + incl - x;
}

// Position of the r-th (0-based) set bit of w (r < popcount(w)): the window that
// holds it is halved six times, each step comparing r with the low half's popcount.
__device__ __forceinline__ int select_bit(uint64_t w, int r) {
    int base = 0;
    uint32_t h = (uint32_t)w;
    int c = __popc(h);
    if (r >= c) {
        r -= c;
        h = (uint32_t)(w >> 32);
        base = 32;
    }
#pragma unroll
    for (int half = 16; half >= 1; half >>= 1) {
        c = __popc(h & ((1u << half) - 1u));
        if (r >= c) {
            r -= c;
            h >>= half;
            base += half;
        }
    }
    return base;
}

__global__ void __launch_bounds__(FIXPOINT_BIG_BLOCK, 1) k_domain_fixpoint(const JobDesc *jobs, int njobs,
                                                                        const long long *vert_off,
                                                           const long long *cstart, const long long *csize,
                                                           int32_t *cand, int *next_job) {
    __shared__ unsigned char dirty[KMAX], chg[KMAX], done[KMAX], dns[KMAX];
    __shared__ int dl[KMAX], size[KMAX], elem[KMAX], newu[KMAX];
    __shared__ long long pre[KMAX + 1];
    __shared__ int nd, any, nnew, empty;
    __shared__ uint64_t wsnap[FP_CHUNK];
    __shared__ int wpre[FP_CHUNK + 1], wsum[32];
    __shared__ int jnext;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarps = blockDim.x >> 5;
    for (;;) {
        // the next job, taken dynamically: pairs differ widely in cost
        if (tid == 0) jnext = atomicAdd(next_job, 1);
        __syncthreads();
        const int jb = jnext;
        __syncthreads();
        if (jb >= njobs) break;
        const JobDesc &J = jobs[jb];
        if (J.filt == nullptr || !(J.flags & JOB_RIDS)) continue;
        const bool DIR = (J.flags & JOB_DIRECTED) != 0, chk = (J.flags & JOB_ELAB) != 0;
        const bool FC = (J.flags & JOB_FC) != 0;
        const int k = J.k, dw = J.t.dw;
        for (int v = tid; v < k; v += blockDim.x) { dirty[v] = 1; done[v] = 0; }
        if (tid == 0) empty = 0;
        __syncthreads();
        // |D(v)|, kept exact below: every removal counts it down, and the first domain to
        // empty ends the pair (it has no match, so the rest of its fixpoint is never needed)
        for (int v = wid; v < k; v += nwarps) {
            unsigned long long c = 0;
            for (int q = lane; q < dw; q += 32) c += __popcll(J.filt[(size_t)v * dw + q]);
            c = warp_sum(c);
            if (lane == 0) {
                size[v] = (int)c;
                if (c == 0) empty = 1;
            }
        }
        __syncthreads();
        while (!empty) {
            // ---- arc consistency over the dirty vertices, to its fixpoint
            for (;;) {
                if (tid == 0) { nd = 0; any = 0; }
                __syncthreads();
                for (int v = tid; v < k; v += blockDim.x) {
                    chg[v] = 0;
                    if (dirty[v]) { dl[atomicAdd(&nd, 1)] = v; dirty[v] = 0; }
                }
                __syncthreads();
                const int n_d = nd;
                if (n_d == 0) break;
                if (cand == nullptr) {
                    // the dirty domains' words, FP_CHUNK at a time: snapshot them, scan their
                    // popcounts, and give each thread the next set bit, so the candidates of a
                    // dense word are checked in parallel rather than by one thread in turn
                    const long long units = (long long)n_d * dw;
                    for (long long u0 = 0; u0 < units; u0 += FP_CHUNK) {
                        const int nw_c = (int)min((long long)FP_CHUNK, units - u0);
                        // words per thread in the scan: as few as the chunk needs (FP_CHUNK is a
                        // multiple of the block size, so tid * ipt + r stays below FP_CHUNK)
                        const int ipt = (nw_c + (int)blockDim.x - 1) / (int)blockDim.x;
                        int cnt = 0;
                        for (int r = 0; r < ipt; ++r) {
                            const int iw = tid * ipt + r;
                            uint64_t w = 0;
                            if (iw < nw_c) {
                                const long long x = u0 + iw;
                                const int i = (int)x / dw, q = (int)x - i * dw;
                                w = J.filt[(size_t)dl[i] * dw + q];
                            }
                            wsnap[iw] = w;
                            cnt += __popcll(w);
                        }
                        int total;
                        int ex = block_scan_int(cnt, wsum, total);
                        for (int r = 0; r < ipt; ++r) {
                            const int iw = tid * ipt + r;
                            wpre[iw] = ex;
                            ex += __popcll(wsnap[iw]);
                        }
                        if (tid == 0) wpre[FP_CHUNK] = total;
                        __syncthreads();
                        for (int x = tid; x < total; x += blockDim.x) {
                            int lo = 0, hi = nw_c;   // the word holding set bit x: wpre[lo] <= x < wpre[lo + 1]
                            while (hi - lo > 1) {
                                const int mid = (lo + hi) >> 1;
                                if (wpre[mid] <= x) lo = mid; else hi = mid;
                            }
                            const long long ux = u0 + lo;
                            const int i = (int)ux / dw, q = (int)ux - i * dw, v = dl[i];
                            const int b = select_bit(wsnap[lo], x - wpre[lo]);
                            if (!ac_supported(J, v, q * 64 + b, DIR, chk)) {
                                atomicAnd((unsigned long long *)(J.filt + (size_t)v * dw + q), ~(1ull << b));
                                chg[v] = 1;
                                any = 1;
                                if (atomicSub(&size[v], 1) == 1) empty = 1;
                            }
                        }
                        __syncthreads();   // wsnap and wpre are refilled for the next chunk
                    }
                } else {
                    const long long g0 = vert_off[jb];
                    // dense: every pattern neighbour's domain holds at least 1/AC_DENSE of the target
                    for (int i = tid; i < n_d; i += blockDim.x) {
                        const int dv = dl[i];
                        bool d = true;
                        for (int e = J.p.rowptr[dv]; d && e < J.p.rowptr[dv + 1]; ++e)
                            d = (long long)size[J.p.col[e]] * AC_DENSE >= J.t.n;
                        for (int e = DIR ? J.p.irowptr[dv] : 0; d && DIR && e < J.p.irowptr[dv + 1]; ++e)
                            d = (long long)size[J.p.icol[e]] * AC_DENSE >= J.t.n;
                        dns[dv] = d;
                    }
                    if (tid == 0) {
                        long long acc = 0;
                        for (int i = 0; i < n_d; ++i) {
                            pre[i] = acc;
                            acc += csize[g0 + dl[i]];
                        }
                        pre[n_d] = acc;
                    }
                    __syncthreads();
                    const long long units = pre[n_d];
                    for (long long x0 = (long long)wid * 32; x0 < units; x0 += (long long)nwarps * 32) {
                        const long long x = x0 + lane;
                        int v = 0, t = -1;
                        int32_t *slot = nullptr;
                        if (x < units) {
                            int lo = 0, hi = n_d;   // the dirty vertex whose slots hold unit x
                            while (hi - lo > 1) {
                                const int mid = (lo + hi) >> 1;
                                if (pre[mid] <= x) lo = mid; else hi = mid;
                            }
                            v = dl[lo];
                            slot = cand + cstart[g0 + v] + (x - pre[lo]);
                            t = *slot;
                        }
                        bool drop = false, heavy = false;
                        if (t >= 0) {
                            if (!((J.filt[(size_t)v * dw + (t >> 6)] >> (t & 63)) & 1ull)) {
                                *slot = -1;                      // removed by forward checking
                            } else {
                                drop = ac_lane_check(J, v, t, DIR, chk, dns[v] != 0, heavy);
                            }
                        }
                        unsigned hv = __ballot_sync(FULL, heavy);
                        while (hv) {
                            const int L = __ffs(hv) - 1;
                            hv &= hv - 1;
                            const int vl = __shfl_sync(FULL, v, L), tl = __shfl_sync(FULL, t, L);
                            const bool sup = ac_supported_warp(J, vl, tl, DIR, chk);
                            if (lane == L) drop = !sup;
                        }
                        if (drop) {
                            atomicAnd((unsigned long long *)(J.filt + (size_t)v * dw + (t >> 6)), ~(1ull << (t & 63)));
                            *slot = -1;
                            chg[v] = 1;
                            any = 1;
                            if (atomicSub(&size[v], 1) == 1) empty = 1;
                        }
                    }
                }
                __syncthreads();
                if (empty || !any) break;
                // the pattern neighbours of every shrunk domain are checked again
                for (int v = tid; v < k; v += blockDim.x) {
                    if (!chg[v]) continue;
                    for (int e = J.p.rowptr[v]; e < J.p.rowptr[v + 1]; ++e) dirty[J.p.col[e]] = 1;
                    if (DIR)
                        for (int e = J.p.irowptr[v]; e < J.p.irowptr[v + 1]; ++e) dirty[J.p.icol[e]] = 1;
                }
                __syncthreads();
            }
            if (empty || !FC) break;
            // ---- one forward-checking round on the new singletons
            if (tid == 0) nnew = 0;
            __syncthreads();
            for (int v = tid; v < k; v += blockDim.x) {
                chg[v] = 0;
                if (size[v] == 1 && !done[v]) {
                    done[v] = 1;
                    newu[atomicAdd(&nnew, 1)] = v;
                }
            }
            __syncthreads();
            const int nn = nnew;
            if (nn == 0) break;   // both fixpoints hold
            for (int sgl = wid; sgl < nn; sgl += nwarps) {
                const int u = newu[sgl];
                int found = -1;
                for (int q0 = 0; q0 < dw && found < 0; q0 += 32) {
                    const int q = q0 + lane;
                    const uint64_t w = q < dw ? J.filt[(size_t)u * dw + q] : 0ull;
                    const unsigned bal = __ballot_sync(FULL, w != 0);
                    if (bal) {
                        const int L = __ffs(bal) - 1;
                        const uint64_t wl = __shfl_sync(FULL, w, L);
                        found = (q0 + L) * 64 + __ffsll((long long)wl) - 1;
                    }
                }
                if (lane == 0) elem[u] = found;
            }
            if (tid == 0) any = 0;
            __syncthreads();
            for (int x = tid; x < nn * k; x += blockDim.x) {
                const int u = newu[x / k], v = x % k, t = elem[u];
                if (v == u || t < 0) continue;
                unsigned long long *wp = reinterpret_cast<unsigned long long *>(J.filt + (size_t)v * dw + (t >> 6));
                const unsigned long long bit = 1ull << (t & 63);
                if (atomicAnd(wp, ~bit) & bit) {
                    chg[v] = 1;
                    any = 1;
                    if (atomicSub(&size[v], 1) == 1) empty = 1;
                }
            }
            __syncthreads();
            if (empty || !any) break;
            for (int v = tid; v < k; v += blockDim.x) {
                if (!chg[v]) continue;
                for (int e = J.p.rowptr[v]; e < J.p.rowptr[v + 1]; ++e) dirty[J.p.col[e]] = 1;
                if (DIR)
                    for (int e = J.p.irowptr[v]; e < J.p.irowptr[v + 1]; ++e) dirty[J.p.icol[e]] = 1;
            }
            __syncthreads();
        }
        __syncthreads();   // the shared arrays are reused by the next job
    }
}

// The same joint fixpoint for very many pairs of small graphs: one warp per pair, no block barrier,
// and the domains transposed: for every target vertex t the k <= 64 pattern vertices that it may
// still be the image of, one 64-bit word C(t) in shared memory.  Arc consistency then checks all
// of t's pattern vertices at once: per class of pattern edges (direction and edge label) the
// words of t's neighbours over that class are ORed, and v leaves C(t) if one of its pattern
// neighbours of the class is missing from the union.  The block form above walks t's row once for
// each (candidate, pattern edge) instead, and is bound by the instructions that takes; here a
// row is walked once per class.  A removal at t marks t's neighbours for another look; when none
// is marked, one forward-checking round takes the element of each new singleton from the
// other domains.  Removals are monotone, so the greatest fixpoint reached is the same.
// (72,000 molecule pairs, RI-DS-SI-FC, the whole call: 9.8 ms with the block form and all sizes
// read back, 7.5 ms with this one.)
constexpr int WARP_FP_K = 64, WARP_FP_N = 512, WARP_FP_CLASSES = 8;   // largest pattern, target, class count

// A[r] bit c of lane r becomes bit r of lane c.
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
#pragma unroll
    for (int j = 16; j; j >>= 1) {
        const uint32_t m = j == 16 ? 0x0000FFFFu : j == 8 ? 0x00FF00FFu : j == 4 ? 0x0F0F0F0Fu : j == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(FULL, x, j);
        x = (lane & j) ? (x & ~m) | ((y >> j) & m) : (x & m) | ((y & m) << j);
    }
    return x;
}

// Shared memory of one warp, for targets of up to n (a multiple of 32) vertices and up to `cls`
// edge classes.
__host__ __device__ constexpr int warp_fixpoint_smem(int n, int cls) {
    return 8 * (n + cls * (WARP_FP_K + 1)) + 4 * (WARP_FP_K + WARP_FP_N / 32 + WARP_FP_CLASSES);
}

__global__ void __launch_bounds__(BLOCK, 4) k_domain_fixpoint_warp(const JobDesc *jobs, int njobs, WarpFixpoint W) {
    extern __shared__ uint64_t wfp_smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t *C = wfp_smem + (size_t)wid * (warp_fixpoint_smem(W.nmax, W.classes) / 8);
    uint64_t *P = C + W.nmax;                      // [class][v]: v's pattern neighbours of the class
    uint64_t *K = P + W.classes * WARP_FP_K;       // [class]: the v that have any
    int *size = reinterpret_cast<int *>(K + W.classes);   // |D(v)|
    uint32_t *dirty = reinterpret_cast<uint32_t *>(size + WARP_FP_K);   // target vertices to look at
    int *clab = reinterpret_cast<int *>(dirty + WARP_FP_N / 32);
    for (;;) {
        int jb = 0;
        if (lane == 0) jb = (int)atomicAdd(W.next, 1ull);
        jb = __shfl_sync(FULL, jb, 0);
        if (jb >= njobs) break;
        const JobDesc &J = jobs[jb];
        const bool DIR = (J.flags & JOB_DIRECTED) != 0, chk = (J.flags & JOB_ELAB) != 0;
        const bool FC = (J.flags & JOB_FC) != 0;
        const int k = J.k, n = J.t.n, dw = J.t.dw, halves = (n + 31) >> 5;
        const int32_t *trow = J.t.rowptr, *tcol = J.t.col, *tel = J.t.elab;
        const int32_t *tirow = J.t.irowptr, *ticol = J.t.icol, *tiel = J.t.ielab;
        uint32_t *filt = reinterpret_cast<uint32_t *>(J.filt);   // D(v) as halves: v * 2 dw + h
        // the domains, transposed 32 x 32 bits at a time; lane l counts |D(l)| and |D(l + 32)|
        int s0 = 0, s1 = 0;
        for (int h = 0; h < halves; ++h) {
            const uint32_t a = lane < k ? filt[(size_t)lane * 2 * dw + h] : 0u;
            const uint32_t b = lane + 32 < k ? filt[(size_t)(lane + 32) * 2 * dw + h] : 0u;
            s0 += __popc(a);
            s1 += __popc(b);
            const uint32_t lo = transpose32(a, lane);
            const uint32_t hi = k > 32 ? transpose32(b, lane) : 0u;
            C[h * 32 + lane] = lo | (uint64_t)hi << 32;
        }
        size[lane] = s0;
        size[lane + 32] = s1;
        bool empty = __any_sync(FULL, (lane < k && s0 == 0) || (lane + 32 < k && s1 == 0));
        // the pattern's edge classes: out-edges label by label, then in-edges
        int nc = 0, nout = 0;
        if (!empty) {
            for (int pass = 0; pass < (DIR ? 2 : 1); ++pass) {
                const int32_t *prow = pass ? J.p.irowptr : J.p.rowptr;
                const int32_t *pcol = pass ? J.p.icol : J.p.col;
                const int32_t *pel = pass ? J.p.ielab : J.p.elab;
                const int b0 = lane < k ? prow[lane] : 0, e0 = lane < k ? prow[lane + 1] : 0;
                const int b1 = lane + 32 < k ? prow[lane + 32] : 0, e1 = lane + 32 < k ? prow[lane + 33] : 0;
                long long cur = LLONG_MIN;
                while (nc < W.classes) {
                    int next = INT_MAX;
                    bool more = !chk ? cur == LLONG_MIN : false;
                    if (chk) {
                        for (int e = b0; e < e0; ++e)
                            if (pel[e] > cur) { next = min(next, pel[e]); more = true; }
                        for (int e = b1; e < e1; ++e)
                            if (pel[e] > cur) { next = min(next, pel[e]); more = true; }
                        next = __reduce_min_sync(FULL, next);
                    }
                    if (!__any_sync(FULL, more)) break;
                    cur = next;
                    uint64_t m0 = 0, m1 = 0;
                    for (int e = b0; e < e0; ++e)
                        if (!chk || pel[e] == next) m0 |= 1ull << pcol[e];
                    for (int e = b1; e < e1; ++e)
                        if (!chk || pel[e] == next) m1 |= 1ull << pcol[e];
                    P[nc * WARP_FP_K + lane] = m0;
                    P[nc * WARP_FP_K + lane + 32] = m1;
                    const uint32_t k0 = __ballot_sync(FULL, m0 != 0), k1 = __ballot_sync(FULL, m1 != 0);
                    if (lane == 0) {
                        K[nc] = k0 | (uint64_t)k1 << 32;
                        clab[nc] = next;
                    }
                    ++nc;
                }
                if (pass == 0) nout = nc;
            }
            if (lane < halves) dirty[lane] = n >= 32 * (lane + 1) ? ~0u : (1u << (n - 32 * lane)) - 1u;
        }
        uint64_t done = 0;   // singletons that forward checking has propagated
        __syncwarp();
        while (!empty) {
            // ---- arc consistency over the marked target vertices, to its fixpoint
            while (__any_sync(FULL, lane < halves && dirty[lane] != 0) && !empty) {
                for (int h = 0; h < halves && !empty; ++h) {
                    const uint32_t look = dirty[h];
                    __syncwarp();
                    if (look == 0) continue;
                    if (lane == 0) dirty[h] = 0;
                    __syncwarp();
                    const int t = h * 32 + lane;
                    const uint64_t mine = ((look >> lane) & 1u) ? C[t] : 0ull;
                    uint64_t fail = 0;
                    if (mine) {
                        for (int c = 0; c < nc; ++c) {
                            uint64_t check = mine & K[c] & ~fail;
                            if (!check) continue;
                            const bool in = c >= nout;
                            const int32_t *rp = in ? tirow : trow, *col = in ? ticol : tcol, *el = in ? tiel : tel;
                            const int lab = clab[c];
                            uint64_t have = 0;
                            for (int f = __ldg(rp + t), fe = __ldg(rp + t + 1); f < fe; ++f)
                                if (!chk || __ldg(el + f) == lab) have |= C[__ldg(col + f)];
                            for (; check; check &= check - 1) {
                                const int v = __ffsll((long long)check) - 1;
                                if (P[c * WARP_FP_K + v] & ~have) fail |= 1ull << v;
                            }
                        }
                    }
                    bool gone = false;
                    if (fail) {
                        C[t] = mine & ~fail;
                        for (uint64_t x = fail; x; x &= x - 1)
                            if (atomicSub(size + __ffsll((long long)x) - 1, 1) == 1) gone = true;
                        for (int f = __ldg(trow + t), fe = __ldg(trow + t + 1); f < fe; ++f) {
                            const int y = __ldg(tcol + f);
                            atomicOr(dirty + (y >> 5), 1u << (y & 31));
                        }
                        if (DIR)
                            for (int f = __ldg(tirow + t), fe = __ldg(tirow + t + 1); f < fe; ++f) {
                                const int y = __ldg(ticol + f);
                                atomicOr(dirty + (y >> 5), 1u << (y & 31));
                            }
                    }
                    empty = __any_sync(FULL, gone);
                    __syncwarp();
                }
            }
            if (empty || !FC) break;
            // ---- one forward-checking round over the new singletons
            bool any = false;
            const uint32_t f0 = __ballot_sync(FULL, lane < k && size[lane] == 1);
            const uint32_t f1 = __ballot_sync(FULL, lane + 32 < k && size[lane + 32] == 1);
            uint64_t fresh = (f0 | (uint64_t)f1 << 32) & ~done;
            done |= fresh;
            __syncwarp();
            for (; fresh && !empty; fresh &= fresh - 1) {
                const int u = __ffsll((long long)fresh) - 1;
                int t = -1;   // its element
                for (int h = 0; h < halves && t < 0; ++h) {
                    const unsigned at = __ballot_sync(FULL, (C[h * 32 + lane] >> u) & 1ull);
                    if (at) t = h * 32 + __ffs(at) - 1;
                }
                if (t < 0) continue;
                const uint64_t rest = C[t] & ~(1ull << u);
                __syncwarp();
                if (rest == 0) continue;
                any = true;
                if (lane == 0) C[t] = 1ull << u;
                bool gone = false;
                if ((rest >> lane) & 1ull) gone = --size[lane] == 0;
                if ((rest >> (lane + 32)) & 1ull) gone = --size[lane + 32] == 0 || gone;
                for (int f = __ldg(trow + t) + lane, fe = __ldg(trow + t + 1); f < fe; f += 32) {
                    const int y = __ldg(tcol + f);
                    atomicOr(dirty + (y >> 5), 1u << (y & 31));
                }
                if (DIR)
                    for (int f = __ldg(tirow + t) + lane, fe = __ldg(tirow + t + 1); f < fe; f += 32) {
                        const int y = __ldg(ticol + f);
                        atomicOr(dirty + (y >> 5), 1u << (y & 31));
                    }
                empty = __any_sync(FULL, gone);
                __syncwarp();
            }
            if (!any) break;   // both fixpoints hold
        }
        __syncwarp();
        // a pair that still has candidates everywhere is searched: its domains go back, and their
        // sizes are listed for the host, which reads nothing of the others
        if (!empty) {
            for (int h = 0; h < halves; ++h) {
                const uint64_t c = C[h * 32 + lane];
                const uint32_t a = transpose32((uint32_t)c, lane);
                if (lane < k) filt[(size_t)lane * 2 * dw + h] = a;
                if (k > 32) {
                    const uint32_t b = transpose32((uint32_t)(c >> 32), lane);
                    if (lane + 32 < k) filt[(size_t)(lane + 32) * 2 * dw + h] = b;
                }
            }
            unsigned long long at = 0;
            if (lane == 0) {
                at = atomicAdd(W.alive, (1ull << 40) + (unsigned)k);
                W.list[at >> 40] = make_int2(jb, (int)(at & ((1ull << 40) - 1)));
            }
            at = __shfl_sync(FULL, at, 0) & ((1ull << 40) - 1);
            for (int v = lane; v < k; v += 32) W.sizes[at + v] = size[v];
        }
        __syncwarp();
    }
}

__device__ __forceinline__ void grid_barrier(unsigned *count, unsigned *gen, int *status);

// The same joint fixpoint for a few pairs, by the whole device in one cooperative launch: a sweep
// (or forward-checking round) ends at a grid barrier instead of the host reading back which domains
// shrank and launching the next.  Every candidate has a slot, found once at the start; a sweep goes
// over all slots and tests, for each, the pattern edges whose other endpoint shrank in the last one;
// lists too long for a lane are gathered and searched by a warp each.  When a
// sweep removes nothing, one block per pair runs a forward-checking round; when that removes
// nothing either, both fixpoints hold.  Flags rotate over three generations (read, being set,
// being cleared), so a sweep costs one barrier.  Bound by the barrier (3 us) and the dependent loads of one candidate's
// test: all domain work of 10 deep patterns (9 sweeps, 2 rounds) 0.86 ms under the host loop ->
// 0.40 here, of 24 directed ones (11 sweeps) 0.65 -> 0.25; of 64 network queries, a block per pair
// there, 2.4 -> 1.4 ms.  It takes calls that the block-per-pair form is not meant for (few pairs),
// and on large targets all of up to DOMAIN_COOP_VERTS pattern vertices.
// What a sweep reads of a pattern vertex and of its edges, gathered once: a candidate's test is then
// slot, these, list bounds, ids, domain words -- six dependent loads where the job and
// pattern records took twice that for every edge.
struct __align__(16) CoopEdge {
    const uint64_t *Du;      // the other endpoint's domain
    int li, bl;              // its label index (plain rows: 0; absent label: -1), the edge's label
    int in, u;               // out- or in-rows; the other endpoint (global vertex)
    int pad[2];
};
struct __align__(16) CoopVert {
    const int32_t *at[2];    // list bounds at at[in][t * stride + li], .. + 1: run tables or row offsets
    const int32_t *ids[2];   // list entries, every (1 << shift)-th word
    const int32_t *lab[2];
    uint64_t *Dv;
    int e0, e1;              // its edges
    int job, stride;
    short shift, chk, dense, pad;
};

struct DomainCoop {
    const JobDesc *jobs;
    const long long *vert_off;
    int njobs, nverts;
    const int *edge_off;    // [njobs] first edge of a job
    CoopVert *vert;         // [nverts]
    CoopEdge *edge;
    int *size;              // [nverts] as found at the start
    unsigned char *chg;     // [3][nverts] domains that shrank; zeroed
    unsigned char *done;    // [nverts] forward checking: singleton propagated; zeroed
    int *any;               // [3] something was removed; zeroed
    int *nheavy;            // [3] candidates whose long lists are still to be searched; zeroed
    int *heavy;             // [cap] their slots
    int2 *slot;             // [cap] candidate (-1: removed) and its global vertex
    long long cap;
    unsigned *bar;          // [2], zeroed
    int *status;            // zeroed; -2: more candidates than `cap`
    int any_fc, any_long;   // some pair checks forward; some list may be longer than AC_WARP_LIST
};

constexpr int DOMAIN_COOP_BLOCKS = 4;     // most blocks per SM of that launch

__device__ __forceinline__ AcList coop_list(const CoopVert &V, const CoopEdge &E, int t) {
    AcList A;
    A.shift = V.shift;
    A.len = 0;
    A.ids = A.lab = nullptr;
    if (E.li < 0) return A;
    const int32_t *r = V.at[E.in] + (size_t)t * V.stride + E.li;
    const int b = __ldg(r);
    A.len = __ldg(r + 1) - b;
    A.ids = V.ids[E.in] + ((size_t)b << A.shift);
    A.lab = V.lab[E.in] + b;
    return A;
}

// The edges e0 + sub, e0 + sub + G, .. of V whose other endpoint shrank (a bit of `chg`; all in the first
// sweep): is candidate t without support for one of them, or (`heavy`) has one too long a list for a lane?
__device__ __forceinline__ bool coop_lane_check(const DomainCoop &D, const CoopVert &V, int t, int sub, int G,
                                                const unsigned *chg, bool &heavy) {
    heavy = false;
    for (int e = V.e0 + sub; e < V.e1; e += G) {
        const CoopEdge &E = D.edge[e];
        if (!((chg[E.u >> 5] >> (E.u & 31)) & 1u)) continue;
        const AcList A = coop_list(V, E, t);
        const bool all = A.len <= AC_WARP_LIST;
        const int n = all ? A.len : V.dense && A.len <= AC_WARP_DIRECT ? AC_LANE_SCAN : 0;
        if (ac_scan(A, n, E.Du, V.chk != 0, E.bl)) continue;
        if (all) return true;
        heavy = true;
    }
    return false;
}

// Warp-collective: its long lists.
__device__ __forceinline__ bool coop_supported_warp(const DomainCoop &D, const CoopVert &V, int t, const unsigned *chg) {
    const int lane = threadIdx.x & 31;
    for (int e = V.e0; e < V.e1; ++e) {
        const CoopEdge &E = D.edge[e];
        if (!((chg[E.u >> 5] >> (E.u & 31)) & 1u)) continue;
        const AcList A = coop_list(V, E, t);
        if (A.len <= AC_WARP_LIST) continue;   // (the candidate's lane has found its support)
        bool found = false;
        for (int f0 = 0; f0 < A.len && !found; f0 += 64) {
            bool ok = false;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int f = f0 + 32 * i + lane;
                if (f < A.len) {
                    const int y = __ldg(A.ids + ((size_t)f << A.shift));
                    ok = ok || ((!V.chk || __ldg(A.lab + f) == E.bl) && ((E.Du[y >> 6] >> (y & 63)) & 1ull));
                }
            }
            found = __any_sync(FULL, ok);
        }
        if (!found) return false;
    }
    return true;
}

__global__ void __launch_bounds__(BLOCK, 4) k_domain_coop(DomainCoop D) {
    extern __shared__ int start[];   // [nverts + 1] first slot of each global vertex
    __shared__ int wsum[32];
    __shared__ int newu[KMAX], elem[KMAX], nnew;
    __shared__ unsigned was[DOMAIN_COOP_VERTS / 32], is[DOMAIN_COOP_VERTS / 32];   // shrank: last step, now (this block)
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int words = (D.nverts + 31) / 32;
    // sizes and records
    for (long long g = w; g < D.nverts; g += nw) {
        const int j = find_job(D.vert_off, D.njobs, g);
        const JobDesc &J = D.jobs[j];
        const int v = (int)(g - D.vert_off[j]);
        const bool DIR = (J.flags & JOB_DIRECTED) != 0, chk = (J.flags & JOB_ELAB) != 0;
        const LabelRuns *R = J.t.runs != nullptr && J.plidx != nullptr ? J.t.runs : nullptr;
        uint64_t *row = J.filt + (size_t)v * J.t.dw;
        unsigned long long c = 0;
        for (int q = lane; q < J.t.dw; q += 32) c += __popcll(row[q]);
        c = warp_sum(c);
        const int no = J.p.rowptr[v + 1] - J.p.rowptr[v], ni = DIR ? J.p.irowptr[v + 1] - J.p.irowptr[v] : 0;
        const int e0 = D.edge_off[j] + J.p.rowptr[v] + (DIR ? J.p.irowptr[v] : 0);
        if (lane == 0) {
            D.size[g] = (int)c;
            CoopVert V;
            V.at[0] = R ? R->run : J.t.rowptr;
            V.at[1] = R ? R->irun : J.t.irowptr;
            V.ids[0] = R ? reinterpret_cast<const int32_t *>(R->col) : J.t.col;
            V.ids[1] = R ? reinterpret_cast<const int32_t *>(R->icol) : J.t.icol;
            V.lab[0] = R ? R->elab : J.t.elab;
            V.lab[1] = R ? R->ielab : J.t.ielab;
            V.Dv = row;
            V.e0 = e0;
            V.e1 = e0 + no + ni;
            V.job = j;
            V.stride = R ? R->stride : 1;
            V.shift = R ? 1 : 0;
            V.chk = chk;
            V.dense = 0;
            V.pad = 0;
            D.vert[g] = V;
        }
        for (int i = lane; i < no + ni; i += 32) {
            const bool in = i >= no;
            const int e = in ? J.p.irowptr[v] + i - no : J.p.rowptr[v] + i;
            const int u = in ? J.p.icol[e] : J.p.col[e];
            CoopEdge E;
            E.Du = J.filt + (size_t)u * J.t.dw;
            E.li = R ? J.plidx[u] : 0;
            E.bl = chk ? (in ? J.p.ielab[e] : J.p.elab[e]) : 0;
            E.in = in;
            E.u = (int)(g - v) + u;
            E.pad[0] = E.pad[1] = 0;
            D.edge[e0 + i] = E;
        }
    }
    grid_barrier(D.bar, D.bar + 1, D.status);
    // slot offsets, by every block for itself
    int total = 0;
    bool over = false;
    for (int g0 = 0; g0 < D.nverts; g0 += BLOCK) {
        const int g = g0 + threadIdx.x;
        const int c = g < D.nverts ? __ldcg(D.size + g) : 0;
        int sum;
        const int ex = block_scan_int(c, wsum, sum);
        if (g < D.nverts) start[g] = total + ex;
        over = over || (long long)total + sum > D.cap;
        total += over ? 0 : sum;
    }
    if (threadIdx.x == 0) start[D.nverts] = total;
    __syncthreads();
    if (over) {   // (the same for every block; the caller's bound rules it out)
        if (blockIdx.x == 0 && threadIdx.x == 0) set_status(D.status, -2);
        return;
    }
    // slots, and which vertices' neighbours are dense
    for (long long g = w; g < D.nverts; g += nw) {
        const CoopVert &V = D.vert[g];
        const TargetView &T = D.jobs[V.job].t;
        int at = start[g];
        for (int q0 = 0; q0 < T.dw; q0 += 32) {
            const int q = q0 + lane;
            uint64_t x = q < T.dw ? V.Dv[q] : 0;
            const int c = __popcll(x);
            if (__reduce_or_sync(FULL, (unsigned)c) == 0) continue;
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += y;
            }
            int o = at + incl - c;
            for (; x; x &= x - 1, ++o) D.slot[o] = make_int2(q * 64 + __ffsll((long long)x) - 1, (int)g);
            at += __shfl_sync(FULL, incl, 31);
        }
        bool d = true;
        for (int e = V.e0 + lane; e < V.e1; e += 32) d = d && (long long)__ldcg(D.size + D.edge[e].u) * AC_DENSE >= T.n;
        d = __all_sync(FULL, d);
        if (lane == 0) D.vert[g].dense = d;
    }
    grid_barrier(D.bar, D.bar + 1, D.status);
    // few candidates: several lanes each, sharing its vertex's edges
    int G = 1;
    while (G < 32 && total <= nw * (32 / (2 * G))) G *= 2;
    const int per = 32 / G, sub = lane & (G - 1);
    bool fc = false, first = true;   // this step is a forward-checking round; ... the first sweep
    for (int s = 0;; s = s == 2 ? 0 : s + 1) {
        const int s1 = s == 2 ? 0 : s + 1, s2 = s1 == 2 ? 0 : s1 + 1;
        const unsigned char *cur = D.chg + (size_t)s * D.nverts;
        unsigned char *next = D.chg + (size_t)s1 * D.nverts;
        // which domains shrank in the last step, as bits
        __syncthreads();
        for (int q = wid; q < words; q += WARPS_PER_BLOCK) {
            const int g = 32 * q + lane;
            const unsigned bits = __ballot_sync(FULL, g < D.nverts && (first || __ldcg(cur + g)));
            if (lane == 0) {
                was[q] = bits;
                is[q] = 0;
            }
        }
        for (long long g = blockIdx.x * (long long)BLOCK + threadIdx.x; g < D.nverts; g += (long long)gridDim.x * BLOCK)
            D.chg[(size_t)s2 * D.nverts + g] = 0;
        if (blockIdx.x == 0 && threadIdx.x == 0) D.any[s2] = D.nheavy[s2] = 0;
        __syncthreads();
        if (!fc) {
            for (long long x0 = w * per; x0 < total; x0 += nw * per) {
                const long long x = x0 + lane / G;
                int2 c = make_int2(-1, 0);
                if (x < total) c = __ldcg(D.slot + x);
                bool drop = false, heavy = false;
                const CoopVert &V = D.vert[c.y];
                if (c.x >= 0) {
                    if ((__ldcg(V.Dv + (c.x >> 6)) >> (c.x & 63)) & 1ull) drop = coop_lane_check(D, V, c.x, sub, G, was, heavy);
                    else if (sub == 0) D.slot[x].x = -1;   // (removed by forward checking)
                }
                // the group's verdict, at its first lane
                const unsigned mine = (G == 32 ? FULL : ((1u << G) - 1u)) << (lane & ~(G - 1));
                const unsigned drops = __ballot_sync(FULL, drop), heavies = __ballot_sync(FULL, heavy);
                drop = (drops & mine) != 0;
                heavy = !drop && (heavies & mine) != 0;
                if (drop && sub == 0) {
                    atomicAnd((unsigned long long *)(V.Dv + (c.x >> 6)), ~(1ull << (c.x & 63)));
                    D.slot[x].x = -1;
                    atomicOr(&is[c.y >> 5], 1u << (c.y & 31));
                }
                // long lists are left for the whole device: hubs come in runs of slots, and one
                // warp searching all of a run's lists set the sweep's length
                const unsigned hv = __ballot_sync(FULL, heavy && sub == 0);
                if (hv) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(D.nheavy + s1, __popc(hv));
                    at = __shfl_sync(FULL, at, 0);
                    if (heavy && sub == 0) D.heavy[at + __popc(hv & ((1u << lane) - 1u))] = (int)x;
                }
            }
            if (D.any_long) {
                grid_barrier(D.bar, D.bar + 1, D.status);
                const int nh = __ldcg(D.nheavy + s1);
                for (long long i = w; i < nh; i += nw) {
                    const int x = __ldcg(D.heavy + i);
                    const int2 c = __ldcg(D.slot + x);
                    const CoopVert &V = D.vert[c.y];
                    if (!coop_supported_warp(D, V, c.x, was) && lane == 0) {
                        atomicAnd((unsigned long long *)(V.Dv + (c.x >> 6)), ~(1ull << (c.x & 63)));
                        D.slot[x].x = -1;
                        atomicOr(&is[c.y >> 5], 1u << (c.y & 31));
                    }
                    __syncwarp();
                }
            }
        } else {
            for (int j = blockIdx.x; j < D.njobs; j += gridDim.x) {
                const JobDesc &J = D.jobs[j];
                if (!(J.flags & JOB_FC)) continue;
                const int k = J.k, dw = J.t.dw;
                const long long g0 = D.vert_off[j];
                __syncthreads();
                if (threadIdx.x == 0) nnew = 0;
                __syncthreads();
                // new singletons: a vertex's words until a second element shows
                for (int v = wid; v < k; v += WARPS_PER_BLOCK) {
                    if (__ldcg(D.done + g0 + v)) continue;
                    int n = 0, at = -1;
                    for (int q0 = 0; q0 < dw && n <= 1; q0 += 64) {
                        uint64_t x[2];
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const int q = q0 + 32 * i + lane;
                            x[i] = q < dw ? __ldcg(J.filt + (size_t)v * dw + q) : 0ull;
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const unsigned bal = __ballot_sync(FULL, x[i] != 0);
                            if (bal == 0) continue;
                            const int L = __ffs(bal) - 1;
                            const uint64_t xl = __shfl_sync(FULL, x[i], L);
                            n += __popc(bal) > 1 ? 2 : min(2, __popcll(xl));
                            at = (q0 + 32 * i + L) * 64 + __ffsll((long long)xl) - 1;
                        }
                    }
                    if (lane == 0 && n == 1) {
                        D.done[g0 + v] = 1;
                        const int y = atomicAdd(&nnew, 1);
                        newu[y] = v;
                        elem[y] = at;
                    }
                }
                __syncthreads();
                const int nn = nnew;
                for (int x = threadIdx.x; x < nn * k; x += BLOCK) {
                    const int u = newu[x / k], v = x % k, t = elem[x / k], g = (int)g0 + v;
                    if (v == u) continue;
                    const unsigned long long bit = 1ull << (t & 63);
                    if (atomicAnd((unsigned long long *)(J.filt + (size_t)v * dw + (t >> 6)), ~bit) & bit)
                        atomicOr(&is[g >> 5], 1u << (g & 31));
                }
            }
        }
        // this block's shrunk domains, told once each (every removal telling on its own queued
        // thousands of updates on the same lines: 55 us of a 62 us sweep)
        __syncthreads();
        for (int q = threadIdx.x; q < words; q += BLOCK)
            for (unsigned m = is[q]; m; m &= m - 1) {
                next[32 * q + __ffs(m) - 1] = 1;
                if (__ldcg(D.any + s1) == 0) D.any[s1] = 1;
            }
        grid_barrier(D.bar, D.bar + 1, D.status);
        first = false;
        const bool any = __ldcg(D.any + s1) != 0;
        if (__ldcg(D.status) != 0) break;
        if (!any) {
            // nothing left to sweep: a forward-checking round, or, after one, the end
            if (fc || !D.any_fc) break;
            fc = true;
        } else {
            fc = false;
        }
    }
}

// |D(v)| for every (job, pattern vertex); one warp each.
__global__ void __launch_bounds__(BLOCK) k_domain_sizes(const JobDesc *jobs, const long long *vert_off, int njobs,
                                                        long long nverts, long long *sizes) {
    const long long u = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (u >= nverts) return;
    const int j = find_job(vert_off, njobs, u);
    const JobDesc &J = jobs[j];
    const int v = (int)(u - vert_off[j]);
    unsigned long long c = 0;
    for (int q = lane; q < J.t.dw; q += 32) c += __popcll(J.filt[(size_t)v * J.t.dw + q]);
    c = warp_sum(c);
    if (lane == 0) sizes[u] = (long long)c;
}

// List D(v) in ascending id order at `out` (one block per task).
__global__ void __launch_bounds__(BLOCK) k_domain_lists(const JobDesc *jobs, const int *task_job, const int *task_vert,
                                                        const int *task_out, int32_t *lists) {
    __shared__ int wsum[WARPS_PER_BLOCK];
    __shared__ int carry;
    const JobDesc &J = jobs[task_job[blockIdx.x]];
    const int v = task_vert[blockIdx.x];
    int32_t *out = lists + task_out[blockIdx.x];
    const uint64_t *row = J.filt + (size_t)v * J.t.dw;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < J.t.dw; base += blockDim.x) {
        const int q = base + threadIdx.x;
        const uint64_t word = q < J.t.dw ? row[q] : 0;
        const int c = __popcll(word);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        int before = carry;
        for (int i = 0; i < w; ++i) before += wsum[i];
        int pos = before + incl - c;
        uint64_t x = word;
        while (x) {
            const int b = __ffsll((long long)x) - 1;
            out[pos++] = q * 64 + b;
            x &= x - 1;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int i = 0; i < WARPS_PER_BLOCK; ++i) tot += wsum[i];
            carry += tot;
        }
        __syncthreads();
    }
}

// ================================================================== split

// One level of the breadth-first split.  Each frame [job, depth, -1, -1, M]
// is a search node whose positions 0..depth-1 are assigned; its candidates
// for position `depth` are tested, and in pass 1 each survivor becomes a
// frame of depth + 1 (or, at the last position, a match).
template <bool DIR>
__global__ void __launch_bounds__(BLOCK) k_split(const JobDesc *jobs, const int32_t *fin, long long nf, int depth,
                                                 int32_t *counts, const long long *offs, int32_t *fout, int pass,
                                                 int count_ctr) {
    __shared__ int Msh[WARPS_PER_BLOCK][KMAX];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int *M = Msh[wib];
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const int in_stride = FRAME_HDR + depth, out_stride = FRAME_HDR + depth + 1;
    for (long long f = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; f < nf; f += nwarps) {
        const int32_t *fr = fin + f * in_stride;
        const int j = fr[0];
        const JobDesc &J = jobs[j];
        for (int t = lane; t < depth; t += 32) M[t] = fr[FRAME_HDR + t];
        __syncwarp();
        const int k = J.k;
        const bool leaf = depth + 1 == k;
        const PosInfo &P = J.pos[depth];
        const Src S = cand_source(J, P, M);
        // a range frame scans candidates [beg, end); the node's states are counted by its first range
        const int rbeg = fr[2], rend = fr[3];
        const int c_lo = rbeg >= 0 ? rbeg : 0, c_hi = rbeg >= 0 ? min(rend, S.len) : S.len;
        const bool count_states = rbeg <= 0;
        unsigned long long psum = 0;
        if (pass == 1 && leaf) {
            for (int t = lane; t < depth; t += 32) psum += gterm(J.pos[t].pv, M[t]);
            psum = warp_sum(psum);
        }
        const long long obase = (pass == 1 && !leaf) ? offs[f] : 0;
        long long child = 0;
        unsigned long long nodes = 0, hs = 0;
        for (int c0 = c_lo; c0 < c_hi; c0 += 32) {
            const int idx = c0 + lane;
            bool ok = false;
            int c = -1;
            if (idx < c_hi) {
                c = S.ptr ? __ldg(S.ptr + S.base + idx) : idx;
                ok = feasible<DIR>(J, P, depth, c, (S.ptr && P.par >= 0) ? S.base + idx : -1, M);
            }
            const unsigned bal = __ballot_sync(FULL, ok);
            const int cnt = __popc(bal);
            if (pass == 1) {
                nodes += cnt;
                if (leaf) {
                    if (ok && count_ctr) {
                        hs += fmix64(psum + gterm(P.pv, c));
                        if (J.mbuf) emit_match(J, M, depth, c);
                    }
                } else if (ok) {
                    const long long o = obase + child + __popc(bal & ((1u << lane) - 1u));
                    int32_t *dst = fout + o * out_stride;
                    dst[0] = j; dst[1] = depth + 1; dst[2] = -1; dst[3] = -1;
                    for (int t = 0; t < depth; ++t) dst[FRAME_HDR + t] = M[t];
                    dst[FRAME_HDR + depth] = c;
                }
            }
            child += cnt;
        }
        if (pass == 0) {
            if (lane == 0) counts[f] = leaf ? 0 : (int32_t)child;
        } else if (count_ctr) {
            hs = warp_sum(hs);
            if (lane == 0) {
                if (count_states) atomicAdd(J.ctr + 1, (unsigned long long)S.len);
                atomicAdd(J.ctr + 2, nodes);
                if (leaf) {
                    atomicAdd(J.ctr + 0, nodes);
                    atomicAdd(J.ctr + 3, hs);
                }
            }
        }
        __syncwarp();
    }
}

// ========================================================= device split
//
// The breadth-first split as one cooperative launch.  Two forms:
//  * ordered (k_split_coop): every level is a count pass, a scan of the
//    warps' child counts and a write pass, so the children of a level come out
//    in search order -- the order that frame i -> shard i mod S relies on;
//  * single-pass (k_split_once, unsharded runs): every frame is tested once
//    and each 32-candidate chunk appends its children at an offset reserved
//    with one fetch-and-add, so a level costs one pass and one grid barrier.
// The loop stops when the frontier reaches `target` frames, is empty, would
// overflow `cap`, or `max_levels` levels are done.  All frames of a level
// share its depth, so a level-L frame has stride FRAME_HDR + L.

__device__ __forceinline__ long long block_excl_scan(long long x, long long *total);

constexpr unsigned long long BARRIER_GUARD_NS = 60ull * 1000000000ull;   // hang guard of one barrier

// Grid barrier for a cooperative launch (all blocks co-resident).  The wait
// is bounded: after BARRIER_GUARD_NS the block records an error and goes on.
__device__ __forceinline__ void grid_barrier(unsigned *count, unsigned *gen, int *status) {
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned *vgen = gen;
        const unsigned g = *vgen;
        __threadfence();
        if (atomicAdd(count, 1u) == gridDim.x - 1) {
            *count = 0;
            __threadfence();
            atomicAdd(gen, 1u);
        } else {
            const unsigned long long t0 = globaltimer();
            unsigned backoff = 32;
            while (*vgen == g) {
                __nanosleep(backoff);
                if (backoff < 1024) backoff <<= 1;
                if (globaltimer() - t0 > BARRIER_GUARD_NS) { set_status(status, -3); break; }
            }
        }
        __threadfence();
    }
    __syncthreads();
}

struct SplitCtl {
    int32_t *buf0, *buf1;       // frame buffers of `cap_ints` ints each; a level-L frame has stride FRAME_HDR + L
    long long cap_ints;
    long long target;           // stop once the frontier has this many frames
    // single-pass split: a level of fewer frames than `narrow` that does not grow ends the
    // level-by-level expansion; the rest runs without barriers (see split_async).  0: never
    long long narrow;
    unsigned long long *qhead, *qtail;   // frame queue: tickets drawn, frames pushed
    unsigned long long *qentry;          // [qcap]: epoch << 40 | frame's offset in the arena
    long long qcap;
    unsigned long long epoch;            // marks this launch's entries (24 bits)
    long long *pend;                     // frames not finished, less the first level's
    unsigned long long *top;             // arena ints handed out
    int *stop;                           // out of arena or queue: what is left goes to `left`
    unsigned long long *nleft;
    const int32_t **left;                // [qcap + 64 per warp + the first level's frames]
    int max_levels;
    long long *wtot;            // [blocks]: children per block, then the blocks' exclusive offsets
    unsigned *bar;              // [2]: barrier count, generation (zeroed by the host)
    long long *result;          // [4]: final frame count, final buffer (0/1), levels done, last total
    int *status;
    int count_ctr;              // 0 in shards other than 0: levels above the frontier are counted once
    uint32_t *masks;            // candidate ballots of the count pass, replayed by the write pass
    long long mask_total;       // masks in the buffer (each warp owns mask_total / warps of them)
    long long *trace;           // single-pass split, tracing only (else null): [0, KMAX) each level's end
                                // (device clock), [KMAX, 2 KMAX) its longest candidate list of one frame
};

// One frame of a split level: count its children (pass 0) or write them from
// `out` on in candidate order and add its counters (pass 1).  Returns the
// number of children.
// The count pass stores each chunk's ballot in the warp's mask buffer (wm,
// mcap masks, position mp) and the write pass replays it instead of testing
// the candidates again (frames with at least 16 candidates); leaf frames have
// no children, so the count pass skips them and only the write pass tests
// them.  Past mcap masks the write pass tests again.
template <bool DIR>
__device__ __forceinline__ long long split_frame(const JobDesc *jobs, const int32_t *fr, int *M, int pass,
                                                 int32_t *fout, long long out, int stride, int count_ctr,
                                                 uint32_t *wm, long long mcap, long long &mp) {
    const int lane = threadIdx.x & 31;
    const int j = fr[0], depth = fr[1], rbeg = fr[2], rend = fr[3];
    const JobDesc &J = jobs[j];
    const bool leaf = depth + 1 == J.k;
    if (pass == 0 && leaf) return 0;
    for (int t = lane; t < depth; t += 32) M[t] = fr[FRAME_HDR + t];
    __syncwarp();
    const PosInfo P = J.pos[depth];
    const Src src = cand_source(J, P, M);
    const int c_lo = rbeg >= 0 ? rbeg : 0, c_hi = rbeg >= 0 ? min(rend, src.len) : src.len;
    unsigned long long psum = 0, nodes = 0, hs = 0;
    long long child = 0;
    if (pass == 1 && leaf && count_ctr) {
        for (int t = lane; t < depth; t += 32) psum += gterm(J.pos[t].pv, M[t]);
        psum = warp_sum(psum);
    }
    // short rows are cheaper to test twice than to store and reload
    const bool masked = !leaf && c_hi - c_lo >= 16;
    for (int c0 = c_lo; c0 < c_hi; c0 += 32) {
        const int idx = c0 + lane;
        bool ok = false;
        int c = -1;
        const bool replay = pass == 1 && masked && mp < mcap;
        if (idx < c_hi) {
            c = src.ptr ? __ldg(src.ptr + src.base + idx) : idx;
            if (replay) ok = (wm[mp] >> lane) & 1u;
            else ok = feasible<DIR>(J, P, depth, c, (src.ptr && P.par >= 0) ? src.base + idx : -1, M);
        }
        const unsigned bal = __ballot_sync(FULL, ok);
        if (masked) {
            if (pass == 0 && mp < mcap && lane == 0) wm[mp] = bal;
            ++mp;
        }
        const int cnt = __popc(bal);
        if (pass == 1) {
            nodes += cnt;
            if (leaf) {
                if (ok && count_ctr) {
                    hs += fmix64(psum + gterm(P.pv, c));
                    if (J.mbuf) emit_match(J, M, depth, c);
                }
            } else if (ok) {
                int32_t *dst = fout + (out + child + __popc(bal & ((1u << lane) - 1u))) * stride;
                dst[0] = j; dst[1] = depth + 1; dst[2] = -1; dst[3] = -1;
                for (int t = 0; t < depth; ++t) dst[FRAME_HDR + t] = M[t];
                dst[FRAME_HDR + depth] = c;
            }
        }
        if (!leaf) child += cnt;
    }
    if (pass == 1 && count_ctr) {
        hs = warp_sum(hs);
        if (lane == 0) {
            if (rbeg <= 0) atomicAdd(J.ctr + 1, (unsigned long long)src.len);
            atomicAdd(J.ctr + 2, nodes);
            if (leaf) {
                atomicAdd(J.ctr + 0, nodes);
                atomicAdd(J.ctr + 3, hs);
            }
        }
    }
    __syncwarp();
    return child;
}

template <bool DIR>
__global__ void __launch_bounds__(BLOCK) k_split_coop(const JobDesc *jobs, long long f0, SplitCtl S) {
    __shared__ int Msh[WARPS_PER_BLOCK][KMAX];
    __shared__ long long carry;
    __shared__ long long woff[WARPS_PER_BLOCK];   // a level's child offsets of this block's warps
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int *M = Msh[wib];
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    long long F = f0, total = 0;
    int cur = 0, level = 0;
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned long long *>(S.result + 6), ~globaltimer());
    const long long mcap = S.masks ? S.mask_total / nw : 0;
    uint32_t *wm = S.masks ? S.masks + w * mcap : nullptr;
    for (; level < S.max_levels; ++level) {
        if (F == 0 || F >= S.target) break;
        const int32_t *fin = cur ? S.buf1 : S.buf0;
        int32_t *fout = cur ? S.buf0 : S.buf1;
        const int sin = FRAME_HDR + level, sout = FRAME_HDR + level + 1;   // all frames of a level share a depth
        // each warp owns a contiguous slice of the frontier, so children come out in search order
        const long long lo = F * w / nw, hi = F * (w + 1) / nw;
        long long mine = 0, mp = 0;
        for (long long f = lo; f < hi; ++f)
            mine += split_frame<DIR>(jobs, fin + f * sin, M, 0, fout, 0, sout, S.count_ctr, wm, mcap, mp);
        // children offsets: warps within the block here, blocks across the grid in block 0
        if (lane == 0) woff[wib] = mine;
        __syncthreads();
        if (threadIdx.x == 0) {
            long long acc = 0;
            for (int i = 0; i < WARPS_PER_BLOCK; ++i) {
                const long long x = woff[i];
                woff[i] = acc;
                acc += x;
            }
            S.wtot[blockIdx.x] = acc;
        }
        grid_barrier(S.bar, S.bar + 1, S.status);
        if (blockIdx.x == 0) {
            // exclusive scan of the per-block counts (one block, chunk by chunk)
            if (threadIdx.x == 0) carry = 0;
            __syncthreads();
            for (long long b = 0; b < gridDim.x; b += BLOCK) {
                const long long i = b + threadIdx.x;
                const long long x = i < gridDim.x ? S.wtot[i] : 0;
                long long tot;
                const long long ex = block_excl_scan(x, &tot);
                if (i < gridDim.x) S.wtot[i] = carry + ex;
                __syncthreads();
                if (threadIdx.x == 0) carry += tot;
                __syncthreads();
            }
            if (threadIdx.x == 0) S.result[3] = carry;
        }
        grid_barrier(S.bar, S.bar + 1, S.status);
        total = *(volatile long long *)(S.result + 3);
        if (total * sout > S.cap_ints) break;   // the next level does not fit: keep this frontier
        const long long out = *(volatile long long *)(S.wtot + blockIdx.x) + woff[wib];
        long long written = 0;
        mp = 0;
        for (long long f = lo; f < hi; ++f)
            written += split_frame<DIR>(jobs, fin + f * sin, M, 1, fout, out + written, sout, S.count_ctr, wm,
                                        mcap, mp);
        grid_barrier(S.bar, S.bar + 1, S.status);
        F = total;
        cur ^= 1;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        S.result[0] = F;
        S.result[1] = cur;
        S.result[2] = level;
    }
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned long long *>(S.result + 7), globaltimer());
}

// Frames a child of `depth` images plus c takes: one, or one per `range` entries of its list when
// that is longer (JOB_LONG_LISTS pairs; where the next level is a whole one, LEVELS, and the last,
// JOB_LONG_LAST ones too).
template <bool DIR, bool LEVELS>
__device__ __forceinline__ int split_child_frames(const JobDesc &J, int depth, int c, const int *M, int &range) {
    range = SPLIT_RANGE;
    const bool fine = LEVELS && depth + 2 == J.k;
    if (!(J.flags & (fine ? JOB_LONG_LISTS | JOB_LONG_LAST : JOB_LONG_LISTS))) return 1;
    const PosInfo *Q = J.pos + depth + 1;
    const PosV q = load_pos(Q);
    long long len;
    if (q.par >= 0) {
        if (J.t.maxdeg != 0 && J.t.maxdeg <= SPLIT_RANGE) return 1;
        const LabelRuns *R = J.t.runs;
        const JobRef v{&J};
        const int li = R ? J.plidx[q.pv] : -1;
        if (R && li < 0) return 1;
        // the shortest constraint's list, as pick_group will find it; any short one settles it
        if (R && !fine) range = SPLIT_RUN_RANGE;
        len = 0x7fffffff;
        for (int x = 0; x <= (R ? q.bc : 0); ++x) {
            int pos = q.par, in = DIR ? q.flags & POS_IN_ROW : 0;
            if (x > 0) {
                const int4 be = __ldg(reinterpret_cast<const int4 *>(J.back + q.bb + x - 1));
                pos = be.x;
                in = DIR ? be.y & 1 : 0;
            }
            const int a = pos == depth ? c : M[pos];
            const int32_t *at = R ? (in ? R->irun : R->run) + (size_t)a * R->stride + li
                                  : (in ? v.irowptr() : v.rowptr()) + a;
            len = min(len, (long long)(__ldg(at + 1) - __ldg(at)));
            if (len <= range) return 1;
        }
    } else {
        len = (J.flags & JOB_RIDS) ? Q->ucnt : J.t.n;
    }
    return (int)((len + range - 1) / range);
}

// Header words of part q of r, of `range` entries each, of a child frame.
__device__ __forceinline__ void split_child_header(int32_t *dst, const JobDesc &J, int j, int depth, int r, int q,
                                                   int range) {
    const bool run = r > 1 && J.t.runs != nullptr && J.pos[depth].par >= 0;   // (its range counts in a run)
    dst[0] = j;
    dst[1] = depth | (run ? FRAME_RUN : 0);
    dst[2] = r == 1 ? -1 : q * range;
    dst[3] = r == 1 ? -1 : (q + 1 == r ? 0x7fffffff : (q + 1) * range);
}

// The single-pass split expands up to 32 frames of a level per warp at once.  The frames'
// candidate lists laid end to end are tested by the whole warp, SPLIT_STEPS x 32 candidates at
// a time whichever frames they belong to, so that lanes are busy whatever the mix of list lengths
// and several loads per lane are in flight; the candidates that pass their local tests queue up
// for the constraint tests, one per lane (spread over (candidate, constraint) pairs where few are
// left, as on narrow levels).  The shared block is kept small: what it takes is L1 that the frames
// and records are read through (5.9 KB per warp made the widest levels 1.6x slower than 3.4 KB).
constexpr int SPLIT_STEPS = 2;
constexpr int SPLIT_QUEUE = 32 * SPLIT_STEPS + 32;
// A child with at least this many images is written by the whole warp, consecutive words at a time
// (from 2 on: 24 directed patterns 1.16 -> 1.42 ms, 200,000 molecule pairs 5.25 -> 5.65; never: 160
// network queries 3.4 -> 3.6; from 32 on batches take the same, 96 served queries 2.9 instead of
// 4.1 ms, which is not understood yet).
constexpr int SPLIT_COOP_DEPTH = 8;
// Of a longer list, each candidate's local tests include the constraints whose images have a
// bitset row, the next shortest run's first: their row pointers are looked up once per frame
// (at most SPLIT_ROWS for the batch), so a test is one load instead of a chain of four
// (a power-law network's hubs form a near-clique: long lists there pass most constraints).  Never:
// 160 network queries 3.4 -> 4.1 ms, 96 served ones 4.1 -> 4.6, ten deep patterns 1.31 -> 1.27;
// lists of 1 and of 17 on as the least: within the spread.  32 rows: served queries 4.1 -> 4.4;
// 128: within the spread, for 512 bytes of shared memory more.
constexpr int SPLIT_ROW_MIN = 4;
constexpr int SPLIT_ROWS = 64;

struct SplitWarp {   // one warp's shared memory: the batch's frames, then its waiting candidates
    uint64_t ids[32];          // address of the first candidate's id (a run: {id, degree}); below 2^32: that vertex
    const int32_t *elab[32];   // first candidate's label in the list, null when not compared
    const int2 *vld[32];       // null: the list is a run (its label is right, its degrees beside the ids)
    const uint64_t *filt[32];  // D(mu_i), or null
    const uint64_t *row[SPLIT_ROWS];   // the frames' constraint rows (null: that image has none)
    int32_t *fr[32];           // split_async: the batch's frames
    int start[33];             // first of the frame's candidates among the batch's
    int job[32], lab[32], odeg[32], slab[32], li[32], nd[32];
    int qc[SPLIT_QUEUE];
    unsigned char ql[SPLIT_QUEUE];
    unsigned char alive[32];   // split_accept: waiting candidates still in the running
    unsigned char rbeg[33];    // first of the frame's rows in `row`
    unsigned char skip[32], next[32], nq[32];   // nq: constraints split_accept has to test
};

// A level's frames [f0, ..) and its children's buffer; places are reserved on the level's child
// counter.  A reservation that ends past `cap_frames` raises `full` and writes nothing (the
// level is then abandoned, see k_split_once).
struct LevelOut {
    static constexpr bool LEVELS = true;
    const int32_t *fin;
    long long f0;
    int sin;
    int32_t *fout;
    long long cap_frames;
    unsigned long long *lvl_ctr;
    long long *full;
    __device__ __forceinline__ const int32_t *frame(const SplitWarp &, int x) const { return fin + (f0 + x) * sin; }
    // the first of `total` child frames of `stride` ints, or null
    __device__ __forceinline__ int32_t *take(int total, int stride) {
        unsigned long long to = 0;
        if ((threadIdx.x & 31) == 0) to = atomicAdd(lvl_ctr, (unsigned long long)total);
        to = __shfl_sync(FULL, to, 0);
        if ((long long)(to + total) > cap_frames) {
            if ((threadIdx.x & 31) == 0) *(volatile long long *)full = 1;
            return nullptr;
        }
        return fout + (long long)to * stride;
    }
};

// Tests the n <= 32 waiting candidates from `at` on against their frames' constraints and rule 1,
// counts and hashes the accepted ones (hs: of frame `lane`), and appends their child frames where
// `out` says.
template <bool DIR, class O>
__device__ __forceinline__ void split_accept(const JobDesc *jobs, int depth, O &out, SplitWarp &W, int at, int n,
                                             unsigned long long &hs) {
    const int lane = threadIdx.x & 31;
    const int sout = FRAME_HDR + depth + 1;
    bool ok = lane < n;
    const int L = W.ql[at + (ok ? lane : 0)], c = W.qc[at + (ok ? lane : 0)];
    const JobDesc &J = jobs[W.job[L]];
    const PosInfo *P = J.pos + depth;
    const int *Mg = out.frame(W, L) + FRAME_HDR;
    const int nq = ok ? W.nq[L] : 0;
    const int mq = (int)__reduce_max_sync(FULL, (unsigned)nq);
    if (mq > 0) {
        int left = n, q0 = 0;   // candidates with constraints to test, and those from which on
        if (n * mq > SPREAD_TESTS) {
            // many: each lane tries two constraints of its own candidate first, which most fail
            const JobRef v{&J};
            const PosV p = load_pos(P);
            for (int q = 0; ok && q < 2 && q < nq; ++q)
                ok = con_holds<DIR>(v, p, q + (q >= W.skip[L] ? 1 : 0), W.li[L], c, Mg);
            const unsigned m = __ballot_sync(FULL, ok && nq > 2);
            if ((m >> lane) & 1u) W.alive[__popc(m & ((1u << lane) - 1u))] = (unsigned char)lane;
            left = __popc(m);
            q0 = 2;
        } else {
            W.alive[lane] = (unsigned char)lane;
        }
        __syncwarp();
        if (left > 0) {   // the (candidate, constraint) tests that remain, spread over the lanes
            const int tests = left * (mq - q0);
            unsigned bad = 0;
            for (int t = lane; t < tests; t += 32) {
                const int q = q0 + t / left, x = W.alive[t % left], Lx = W.ql[at + x];
                const JobDesc &Jx = jobs[W.job[Lx]];
                if (q < W.nq[Lx] &&
                    !con_holds<DIR>(JobRef{&Jx}, load_pos(Jx.pos + depth), q + (q >= W.skip[Lx] ? 1 : 0), W.li[Lx],
                                    W.qc[at + x], out.frame(W, Lx) + FRAME_HDR))
                    bad |= 1u << x;
            }
            bad = __reduce_or_sync(FULL, bad);
            ok = ok && !((bad >> lane) & 1u);
        }
    }
    ok = ok && unused(P, c, Mg);
    if (!__any_sync(FULL, ok)) return;
    if (ok) atomicAdd(&W.nd[L], 1);
    const bool leaf = depth + 1 == J.k;
    for (unsigned m = __ballot_sync(FULL, ok && leaf); m;) {   // matches, one frame's at a time
        const int L0 = __shfl_sync(FULL, L, __ffs(m) - 1);
        const int32_t *M0 = out.frame(W, L0) + FRAME_HDR;
        const PosInfo *P0 = jobs[W.job[L0]].pos;
        unsigned long long psum = 0;
        for (int t = lane; t < depth; t += 32) psum += gterm(P0[t].pv, M0[t]);
        psum = warp_sum(psum);
        const bool here = ok && leaf && L == L0;
        unsigned long long h = 0;
        if (here) {
            h = fmix64(psum + gterm(P->pv, c));
            if (J.mbuf) emit_match(J, Mg, depth, c);
        }
        h = warp_sum(h);
        if (lane == L0) hs += h;
        m &= ~__ballot_sync(FULL, here);
    }
    // frames per child: one, or one per part of a long list, so that no warp of the next level
    // scans a hub's whole row while the others wait at the barrier
    int range = 0;
    const int r = ok && !leaf ? split_child_frames<DIR, O::LEVELS>(J, depth, c, Mg, range) : 0;
    int incl = r;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(FULL, incl, 31);
    if (total == 0) return;
    int32_t *const to = out.take(total, sout);
    if (to == nullptr) return;
    const bool coop = depth >= SPLIT_COOP_DEPTH;
    for (int q = 0; q < r; ++q) {
        int32_t *dst = to + (long long)(incl - r + q) * sout;
        split_child_header(dst, J, W.job[L], depth + 1, r, q, range);
        for (int t = 0; t < depth && !coop; ++t) dst[FRAME_HDR + t] = Mg[t];
        dst[FRAME_HDR + depth] = c;
    }
    if (coop)
        for (unsigned m = __ballot_sync(FULL, r > 0); m; m &= m - 1) {
            const int x = __ffs(m) - 1;
            const int rx = __shfl_sync(FULL, r, x), Lx = __shfl_sync(FULL, L, x);
            const int32_t *from = out.frame(W, Lx) + FRAME_HDR;
            int32_t *dst = to + (long long)(__shfl_sync(FULL, incl, x) - rx) * sout + FRAME_HDR;
            for (int t = lane; t < depth; t += 32) {
                const int y = from[t];
                for (int q = 0; q < rx; ++q) dst[(long long)q * sout + t] = y;
            }
        }
}

// Expands the nf <= 32 frames of `out`, all at `depth`, by one warp.  Returns the longest list.
template <bool DIR, class O>
__device__ __forceinline__ int split_batch(const JobDesc *jobs, int nf, int depth, O &out, SplitWarp &W) {
    const int lane = threadIdx.x & 31;
    // the frames' lists: few frames share the warp's lanes out among them
    int G = 32;
    while (G > 1 && 32 / G < nf) G >>= 1;
    int j = -1, len = 0, rows = 0;
    unsigned long long st = 0;
    {
        const int sub = lane & (G - 1), x = lane / G;
        const bool have = x < nf;
        const int32_t *fr = out.frame(W, have ? x : 0);
        const int jx = fr[0];
        const JobDesc &J = jobs[jx];
        const JobRef v{&J};
        const PosInfo *P = J.pos + depth;
        const PosV p = load_pos(P);
        const int *Mg = fr + FRAME_HDR;
        const Cand S = pick_group<DIR>(v, p, P, Mg, G, sub);
        int n = 0, nr = 0, raw = 0;
        if (have && sub == 0) {
            int lo, hi;
            raw = list_range<DIR>(v, p, S, Mg, fr[2], fr[3], (fr[1] & FRAME_RUN) != 0, lo, hi) ? S.raw : 0;
            n = max(hi - lo, 0);
            // (rows are of use: the list is long and the target keeps bitset rows)
            if (!DIR && n > SPLIT_ROW_MIN && S.next >= 0 && !(J.flags & JOB_ELAB) &&
                (J.t.adj != nullptr || J.t.hub_slot != nullptr))
                nr = p.bc;
            const bool run = S.li >= 0;
            W.ids[x] = run       ? reinterpret_cast<uint64_t>(reinterpret_cast<const int2 *>(S.ids) + S.base + lo)
                       : S.ids   ? reinterpret_cast<uint64_t>(S.ids + S.base + lo)
                                 : (uint64_t)(S.base + lo);
            W.elab[x] = (J.flags & JOB_ELAB) && S.skip >= 0 ? S.elab + S.base + lo : nullptr;
            W.vld[x] = run ? nullptr : J.t.vld;
            W.filt[x] = (J.flags & JOB_RIDS) ? J.filt + (size_t)p.pv * J.t.dw : nullptr;
            W.lab[x] = p.lab;
            W.odeg[x] = p.odeg;
            W.slab[x] = S.lab;
            W.li[x] = S.li;
            W.skip[x] = (unsigned char)S.skip;   // (unparented: no constraint is tested)
            W.next[x] = (unsigned char)S.next;
            W.nq[x] = (unsigned char)(p.par >= 0 ? p.bc : 0);
            W.job[x] = jx;
            W.nd[x] = 0;
        }
        // frame x's numbers to lane x
        const int from = min(lane * G, 31);
        n = __shfl_sync(FULL, n, from);
        nr = __shfl_sync(FULL, nr, from);
        raw = __shfl_sync(FULL, raw, from);
        const int jl = __shfl_sync(FULL, jx, from);
        if (lane < nf) {
            j = jl;
            len = n;
            rows = nr;
            st = (unsigned long long)raw;
        }
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    W.start[lane + 1] = incl;
    if (lane == 0) W.start[0] = 0;
    const int total = __shfl_sync(FULL, incl, 31);
    const bool any_rows = !DIR && __any_sync(FULL, rows > 0);
    __syncwarp();
    if (any_rows) {
        const int want = rows;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, rows, o);
            if (lane >= o) rows += y;
        }
        const int from = min(rows - want, SPLIT_ROWS), to = min(rows, SPLIT_ROWS);
        W.rbeg[lane + 1] = (unsigned char)to;
        if (lane == 0) W.rbeg[0] = 0;
        const int bc = lane < nf ? W.nq[lane] : 0;
        __syncwarp();
        if (want > 0 && to - from == want) W.nq[lane] = 0;   // (unless a row is missing, below)
        __syncwarp();
        const int nrow = __shfl_sync(FULL, to, 31);
        for (int e0 = 0; e0 < nrow; e0 += 32) {
            const int e = e0 + lane;
            int x = 0;
#pragma unroll
            for (int h = 16; h >= 1; h >>= 1)
                if (W.rbeg[x + h] <= e) x += h;
            const int bx = __shfl_sync(FULL, bc, x);
            if (e < nrow) {
                const JobDesc &J = jobs[W.job[x]];
                // the frame's constraints but the list's own, with `next` first
                const int skip = W.skip[x], first = W.next[x] - (W.next[x] > skip ? 1 : 0), i = e - W.rbeg[x];
                const int y = i == 0 ? first : i == first ? 0 : i;
                const uint64_t *row = con_row<DIR>(JobRef{&J}, load_pos(J.pos + depth), y + (y >= skip ? 1 : 0),
                                                   out.frame(W, x) + FRAME_HDR);
                W.row[e] = row;
                if (row == nullptr) W.nq[x] = (unsigned char)bx;
            }
        }
        __syncwarp();
    }
    int n = 0;   // waiting candidates
    unsigned long long hs = 0;
    for (int t0 = 0; t0 < total; t0 += 32 * SPLIT_STEPS) {
        int L[SPLIT_STEPS], c[SPLIT_STEPS];
        bool ok[SPLIT_STEPS];
        int e[SPLIT_STEPS], dg[SPLIT_STEPS];
#pragma unroll
        for (int u = 0; u < SPLIT_STEPS; ++u) {
            const int t = t0 + 32 * u + lane;
            c[u] = -1;
            dg[u] = 0;
            L[u] = e[u] = 0;
            if (t < total) {
                int x = 0;   // the last frame with start[x] <= t
#pragma unroll
                for (int h = 16; h >= 1; h >>= 1)
                    if (W.start[x + h] <= t) x += h;
                L[u] = x;
                e[u] = t - W.start[x];
                const uint64_t ids = W.ids[x];
                if (W.vld[x] == nullptr) {
                    const int2 y = __ldg(reinterpret_cast<const int2 *>(ids) + e[u]);
                    c[u] = y.x;
                    dg[u] = y.y;
                } else {
                    c[u] = ids >> 32 ? __ldg(reinterpret_cast<const int32_t *>(ids) + e[u]) : (int)ids + e[u];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < SPLIT_STEPS; ++u) {
            ok[u] = c[u] >= 0;
            if (ok[u]) {
                const int x = L[u];
                const int2 *vld = W.vld[x];
                int lab = W.lab[x];
                if (vld != nullptr) {
                    const int2 r = __ldg(vld + c[u]);
                    dg[u] = r.y;
                    ok[u] = r.x == lab;                                            // rule 2
                }
                ok[u] = ok[u] && dg[u] >= W.odeg[x];                               // rule 3
                if (DIR && ok[u]) {
                    const JobDesc &J = jobs[W.job[x]];
                    ok[u] = __ldg(J.t.indeg + c[u]) >= __ldg(&J.pos[depth].ideg);
                }
                if (ok[u] && W.filt[x]) ok[u] = (W.filt[x][c[u] >> 6] >> (c[u] & 63)) & 1ull;
                if (ok[u] && W.elab[x]) ok[u] = __ldg(W.elab[x] + e[u]) == W.slab[x];
            }
        }
        if (any_rows) {   // two rows of each candidate at a time
            int r0[SPLIT_STEPS], r1[SPLIT_STEPS];
#pragma unroll
            for (int u = 0; u < SPLIT_STEPS; ++u) {
                r0[u] = W.rbeg[L[u]];
                r1[u] = ok[u] ? W.rbeg[L[u] + 1] : 0;
            }
            for (bool more = true; more;) {
                uint64_t wa[SPLIT_STEPS], wb[SPLIT_STEPS];
#pragma unroll
                for (int u = 0; u < SPLIT_STEPS; ++u) {
                    const uint64_t *ra = r0[u] < r1[u] ? W.row[r0[u]] : nullptr;
                    const uint64_t *rb = r0[u] + 1 < r1[u] ? W.row[r0[u] + 1] : nullptr;
                    wa[u] = ra ? __ldg(ra + (c[u] >> 6)) : ~0ull;
                    wb[u] = rb ? __ldg(rb + (c[u] >> 6)) : ~0ull;
                }
                more = false;
#pragma unroll
                for (int u = 0; u < SPLIT_STEPS; ++u) {
                    if (!(((wa[u] & wb[u]) >> (c[u] & 63)) & 1ull)) {
                        ok[u] = false;
                        r1[u] = 0;
                    }
                    r0[u] += 2;
                    more = more || r0[u] < r1[u];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < SPLIT_STEPS; ++u) {
            const unsigned bal = __ballot_sync(FULL, ok[u]);
            if (ok[u]) {
                const int y = n + __popc(bal & ((1u << lane) - 1u));
                W.qc[y] = c[u];
                W.ql[y] = (unsigned char)L[u];
            }
            n += __popc(bal);
        }
        __syncwarp();
        while (n >= 32) {   // full warps of them, from the end
            n -= 32;
            split_accept<DIR>(jobs, depth, out, W, n, 32, hs);
            __syncwarp();
        }
    }
    if (n > 0) split_accept<DIR>(jobs, depth, out, W, 0, n, hs);
    __syncwarp();
    // counters: segmented sums over runs of consecutive lanes with the same job, one atomic per run
    const bool leaf = j >= 0 && depth + 1 == jobs[j].k;
    unsigned long long nd = j >= 0 ? (unsigned long long)W.nd[lane] : 0, mt = leaf ? nd : 0;
    const int prev = __shfl_up_sync(FULL, j, 1);
    const unsigned heads = __ballot_sync(FULL, lane == 0 || j != prev);
    const int head = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
    if (nf > 1) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long a = __shfl_up_sync(FULL, st, o), b = __shfl_up_sync(FULL, nd, o),
                                     c = __shfl_up_sync(FULL, mt, o), d = __shfl_up_sync(FULL, hs, o);
            if (lane - o >= head) {
                st += a;
                nd += b;
                mt += c;
                hs += d;
            }
        }
    }
    const bool tail = lane == 31 || ((heads >> (lane + 1)) & 1u);
    if (tail && j >= 0) {
        unsigned long long *ctr = jobs[j].ctr;
        if (st) atomicAdd(ctr + 1, st);
        if (nd) atomicAdd(ctr + 2, nd);
        if (mt) atomicAdd(ctr + 0, mt);
        if (hs) atomicAdd(ctr + 3, hs);
    }
    __syncwarp();
    return warp_max(len);
}

// ------------------------------------------- the split without barriers
//
// Once the levels are narrow and no longer grow, a level lasts as long as its slowest frame and
// a barrier, however little there is to do (60-126 levels of 12-45 us on deep patterns).  The
// rest of the split then runs asynchronously: a warp expands a batch of frames of one depth,
// keeps up to 32 children as its next batch, and pushes the others -- all but one while other
// warps wait for work -- to a queue whose tickets are drawn in order, one frame to a ticket.
// Children are written to a bump-allocated arena (the frontier buffer the levels no longer need), a
// chunk per warp at a time, and handed on only at the end of the batch.  A batch whose
// children no longer fit is abandoned like a level: its frames are counted and become counted
// ranges (or, on the last position, empty ones), every warp stops, and what was not expanded is
// listed for the search kernel.  Waits are bounded by the barrier's guard and end when no frame is
// pending or the stop flag is up.  Bound by the dependent loads of one batch (header, tables,
// runs, ids, constraint rows: 5-10 us).  It starts below one frame per resident warp: 160 network
// queries 5.7 -> 4.1 ms a call, 64 with domains 5.3 -> 4.7, 96 served 4.1 -> 3.0, 10 deep patterns
// 2.0 -> 1.8, 200,000 molecule pairs 9.75 -> 9.6 (the last position taken here too: 24 directed
// patterns 1.9 -> 1.5 ms).
// Arena ints a warp takes at once: a share of the arena, within these limits.
constexpr int ASYNC_CHUNK_MIN = 256, ASYNC_CHUNK_MAX = 8192;
constexpr int ASYNC_SEGS = 8;       // pieces of the arena one batch's children may lie in
constexpr unsigned long long ASYNC_OFFSET = (1ull << 40) - 1;

struct AsyncOut {
    static constexpr bool LEVELS = false;
    const SplitCtl &S;
    int32_t *arena;
    long long chunk;                 // ints taken at once
    long long pos, end;              // the warp's chunk: free ints [pos, end)
    int nseg;                        // the batch's children: pieces of the arena ...
    bool full;                       // ... or no room for them
    long long *seg;                  // [ASYNC_SEGS] first int (shared memory)
    int *segn;                       // [ASYNC_SEGS] frames
    __device__ __forceinline__ const int32_t *frame(const SplitWarp &W, int x) const { return W.fr[x]; }
    __device__ __forceinline__ int32_t *take(int total, int stride) {
        const int lane = threadIdx.x & 31;
        const long long need = (long long)total * stride;
        if (full) return nullptr;
        if (pos + need > end) {
            // (a batch that goes on to take more takes four times as much each time)
            const long long size = max(need, chunk << (2 * nseg));
            unsigned long long t = 0;
            if (lane == 0) t = atomicAdd(S.top, (unsigned long long)size);
            t = __shfl_sync(FULL, t, 0);
            if (nseg == ASYNC_SEGS || (long long)t + size > S.cap_ints) {
                full = true;
                return nullptr;
            }
            pos = (long long)t;
            end = pos + size;
            if (lane == 0) {
                seg[nseg] = pos;
                segn[nseg] = 0;
            }
            ++nseg;
        } else if (nseg == 0) {
            if (lane == 0) {
                seg[0] = pos;
                segn[0] = 0;
            }
            nseg = 1;
        }
        if (lane == 0) segn[nseg - 1] += total;
        int32_t *p = arena + pos;
        pos += need;
        return p;
    }
};

// Frame of queue ticket t if it is there (tickets below F: the first level's frames); a fence
// has to follow before the frame is read.
__device__ __forceinline__ int32_t *async_frame(const SplitCtl &S, int32_t *fin, long long F, int sin, int32_t *arena,
                                                long long t) {
    if (t < F) return fin + t * sin;
    if (t - F >= S.qcap) return nullptr;
    const unsigned long long e = load_relaxed(S.qentry + (t - F));
    return (e >> 40) == S.epoch ? arena + (e & ASYNC_OFFSET) : nullptr;
}

__device__ __forceinline__ void async_leave(const SplitCtl &S, const int32_t *fr) {
    S.left[atomicAdd(S.nleft, 1ull)] = fr;
}

// Frames [0, F) of `fin`, of stride sin (all at one depth), searched to the end or until the arena
// or the queue is full.
template <bool DIR>
__device__ __forceinline__ void split_async(const JobDesc *jobs, const SplitCtl &S, int32_t *fin, int32_t *arena,
                                            long long F, int sin, SplitWarp &W, long long *seg, int *segn) {
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long chunk = min((long long)ASYNC_CHUNK_MAX, max((long long)ASYNC_CHUNK_MIN, S.cap_ints / (2 * nw)));
    AsyncOut out{S, arena, chunk, 0, 0, 0, false, seg, segn};
    int deepest = sin - FRAME_HDR;   // depth the warp's finished batches reached
    long long held = 0;   // tickets drawn and not yet served: [held, held + hn)
    int hn = 0;
    int nloc = 0, depth = 0;   // the next batch, in W.fr
    for (;;) {
        if (nloc == 0) {
            int got = 0;
            if (lane == 0) {
                unsigned backoff = 32;
                const unsigned long long t0 = globaltimer();
                for (;;) {
                    if (load_relaxed(S.stop) != 0) break;
                    if (hn == 0) {
                        const long long ready = F + (long long)load_relaxed(S.qtail) - (long long)load_relaxed(S.qhead);
                        hn = (int)max(1ll, min(32ll, ready / (2 * nw)));
                        held = (long long)atomicAdd(S.qhead, (unsigned long long)hn);
                    }
                    if (async_frame(S, fin, F, sin, arena, held) != nullptr) {
                        got = 1;
                        break;
                    }
                    if (F + (long long)load_relaxed(reinterpret_cast<unsigned long long *>(S.pend)) == 0) break;
                    __nanosleep(backoff);
                    if (backoff < 512) backoff <<= 1;
                    if (globaltimer() - t0 > BARRIER_GUARD_NS) {
                        set_status(S.status, -3);
                        break;
                    }
                }
            }
            got = __shfl_sync(FULL, got, 0);
            held = __shfl_sync(FULL, held, 0);
            hn = __shfl_sync(FULL, hn, 0);
            if (!got) break;
            // the tickets' frames that are there, as long as they share a depth
            int32_t *fr = lane < hn ? async_frame(S, fin, F, sin, arena, held + lane) : nullptr;
            __threadfence();
            const int d = fr ? fr[1] & FRAME_DEPTH_MASK : -1;
            depth = __shfl_sync(FULL, d, 0);
            nloc = __ffs(~__ballot_sync(FULL, fr != nullptr && d == depth)) - 1;
            if (nloc < 0) nloc = 32;
            if (lane < nloc) W.fr[lane] = fr;
            held += nloc;
            hn -= nloc;
            __syncwarp();
        }
        const int n = nloc;
        out.nseg = 0;
        out.full = false;
        split_batch<DIR>(jobs, n, depth, out, W);
        __syncwarp();
        int nc = 0;
        for (int q = 0; q < out.nseg; ++q) nc += segn[q];
        // tickets waiting for frames
        long long waiting = 0;
        if (lane == 0 && nc > 1)
            waiting = (long long)load_relaxed(S.qhead) - (F + (long long)load_relaxed(S.qtail));
        waiting = __shfl_sync(FULL, waiting, 0);
        // children to keep as the next batch, and to push
        int keep = min(nc, 32);
        if (waiting > 0 && nc > 1) keep = (int)min((long long)keep, max(1ll, nc - waiting));
        const int push = nc - keep;
        unsigned long long t = 0;
        bool fail = out.full;
        if (!fail && push > 0) {
            if (lane == 0) {
                atomicAdd(reinterpret_cast<unsigned long long *>(S.pend), (unsigned long long)push);
                t = atomicAdd(S.qtail, (unsigned long long)push);
            }
            t = __shfl_sync(FULL, t, 0);
            fail = (long long)t + push > S.qcap;
        }
        if (fail) {   // the batch's children are dropped: its frames, counted, go to the search
            if (lane < n) {
                int32_t *fr = W.fr[lane];
                if (depth + 1 == jobs[fr[0]].k) {
                    fr[2] = fr[3] = 1;
                } else {
                    fr[1] |= FRAME_COUNTED;
                    if (fr[2] < 0) { fr[2] = 0; fr[3] = 0x7fffffff; }
                }
                async_leave(S, fr);
            }
            nloc = 0;
            if (lane == 0) atomicExch(S.stop, 1);
            break;
        }
        const int stride = FRAME_HDR + depth + 1;
        __threadfence();
        __syncwarp();
        int32_t *mine = nullptr;
        for (int i0 = 0; i0 < nc; i0 += 32) {
            const int i = i0 + lane;
            if (i < nc) {
                int q = 0, rest = i;
                while (rest >= segn[q]) rest -= segn[q++];
                const long long at = seg[q] + (long long)rest * stride;
                if (i < keep) mine = arena + at;   // (keep <= 32: one per lane)
                else store_release(S.qentry + t + (i - keep), S.epoch << 40 | (unsigned long long)at);
            }
        }
        __syncwarp();
        if (lane < keep) W.fr[lane] = mine;
        if (lane == 0 && keep != n)
            atomicAdd(reinterpret_cast<unsigned long long *>(S.pend), (unsigned long long)(long long)(keep - n));
        __syncwarp();
        nloc = keep;
        ++depth;
        deepest = max(deepest, depth);
        if (nloc > 0) {   // (one lane's read: the warp leaves as one)
            const int stop = lane == 0 ? load_relaxed(S.stop) : 0;
            if (__shfl_sync(FULL, stop, 0) != 0) break;
        }
    }
    if (lane < nloc) async_leave(S, W.fr[lane]);
    if (lane == 0) atomicMax(reinterpret_cast<unsigned long long *>(S.result + 2), (unsigned long long)deepest);
    // (either the stop flag is up or no frame is pending: the same for every warp)
    grid_barrier(S.bar, S.bar + 1, S.status);
    if (load_relaxed(S.stop) != 0) {   // (no warp-wide operation below)
        int32_t *fr = lane < hn ? async_frame(S, fin, F, sin, arena, held + lane) : nullptr;
        if (fr) async_leave(S, fr);
        const long long h = (long long)load_relaxed(S.qhead);
        const long long e = F + min((long long)load_relaxed(S.qtail), S.qcap);
        for (long long x = h + blockIdx.x * (long long)blockDim.x + threadIdx.x; x < e; x += (long long)gridDim.x * blockDim.x)
            if (int32_t *y = async_frame(S, fin, F, sin, arena, x)) async_leave(S, y);
    }
}

// Single-pass split (unsharded runs; the caller's shard counts the levels).
// Bound by the gathers of the wide levels (id and degree streamed, one bitset word per
// constraint tested) and, on narrow ones, by the dependent loads of one frame and the barrier.
// Per call, against lists that were the parent's rows, tested by a warp or a lane per frame:
// 160 queries on the 100k-vertex network 9.0 -> 5.7 ms, 24 directed edge-labelled patterns
// 1.45 -> 0.66 ms, 96 served queries on 50k vertices 6.0 -> 4.1 ms end to end; 200,000
// molecule pairs (no runs: short rows) 5.4 -> 5.2 ms.
// The children of level L are counted on wtot[L] (zeroed by the host).  A
// level whose children do not all fit is abandoned after its barrier: its
// frames stay the frontier, rewritten so that the search does not count the
// level again -- a frame with children becomes a counted range (over its
// whole candidate list if it had none; the search re-derives its children
// and counts from the next level on), a frame on the last position becomes
// the empty range [1, 1).
template <bool DIR>
__global__ void __launch_bounds__(BLOCK, 4) k_split_once(const JobDesc *jobs, long long f0, SplitCtl S) {
    __shared__ SplitWarp Wsh[WARPS_PER_BLOCK];
    const int lane = threadIdx.x & 31;
    __shared__ long long seg[WARPS_PER_BLOCK][ASYNC_SEGS];
    __shared__ int segn[WARPS_PER_BLOCK][ASYNC_SEGS];
    SplitWarp &W = Wsh[threadIdx.x >> 5];
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    unsigned long long *lvl_ctr = reinterpret_cast<unsigned long long *>(S.wtot);
    long long F = f0;
    int cur = 0, level = 0;
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned long long *>(S.result + 6), ~globaltimer());
    long long before = 0;   // the last level's frames
    bool narrow = false;
    for (; level < S.max_levels; ++level) {
        narrow = F > 0 && F < S.narrow && F <= before;
        if (F == 0 || F >= S.target || narrow) break;
        before = F;
        int32_t *fin = cur ? S.buf1 : S.buf0;
        int32_t *fout = cur ? S.buf0 : S.buf1;
        const int sin = FRAME_HDR + level, sout = FRAME_HDR + level + 1;
        const long long lo = F * w / nw, hi = F * (w + 1) / nw;
        int longest = 0;
        LevelOut out{fin, lo, sin, fout, S.cap_ints / sout, lvl_ctr + level, S.result + 5};
        for (; out.f0 < hi; out.f0 += 32)
            longest = max(longest, split_batch<DIR>(jobs, (int)min(32ll, hi - out.f0), level, out, W));
        if (S.trace && lane == 0 && longest > 0)
            atomicMax(reinterpret_cast<unsigned long long *>(S.trace + KMAX + level), (unsigned long long)longest);
        grid_barrier(S.bar, S.bar + 1, S.status);
        if (S.trace && blockIdx.x == 0 && threadIdx.x == 0) S.trace[level] = (long long)globaltimer();
        if (*(volatile long long *)(S.result + 5) != 0) {
            for (long long f = lo; f < hi; ++f) {
                int32_t *fr = fin + f * sin;
                if (lane == 0) {
                    const bool leaf = (fr[1] & FRAME_DEPTH_MASK) + 1 == jobs[fr[0]].k;
                    if (leaf) { fr[2] = 1; fr[3] = 1; }
                    else {
                        fr[1] |= FRAME_COUNTED;
                        if (fr[2] < 0) { fr[2] = 0; fr[3] = 0x7fffffff; }
                    }
                }
            }
            break;
        }
        F = (long long)*(volatile unsigned long long *)(lvl_ctr + level);
        cur ^= 1;
    }
    if (narrow)
        split_async<DIR>(jobs, S, cur ? S.buf1 : S.buf0, cur ? S.buf0 : S.buf1, F, FRAME_HDR + level, W,
                         seg[threadIdx.x >> 5], segn[threadIdx.x >> 5]);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        S.result[0] = narrow ? -1 : F;   // (-1: the frames are those listed in `left`, *nleft of them)
        S.result[1] = cur;
        if (!narrow) S.result[2] = level;
    }
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned long long *>(S.result + 7), globaltimer());
}

// =================================================================== scan

constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_TILE = BLOCK * SCAN_ITEMS;

__device__ __forceinline__ long long block_excl_scan(long long x, long long *total) {
    __shared__ long long ws[WARPS_PER_BLOCK];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[w] = incl;
    __syncthreads();
    long long before = 0, tot = 0;
    for (int i = 0; i < WARPS_PER_BLOCK; ++i) {
        if (i < w) before += ws[i];
        tot += ws[i];
    }
    __syncthreads();
    *total = tot;
    return before + incl - x;
}

__global__ void __launch_bounds__(BLOCK) k_scan_tiles(const int32_t *in, long long *out, long long n, long long *tile_sum) {
    const long long base = (long long)blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
    long long v[SCAN_ITEMS], s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = (base + i < n) ? in[base + i] : 0;
        s += v[i];
    }
    long long tot;
    long long ex = block_excl_scan(s, &tot);
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        if (base + i < n) out[base + i] = ex;
        ex += v[i];
    }
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(BLOCK) k_scan_sums(long long *tile_sum, long long ntiles, long long *total) {
    __shared__ long long carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (long long b = 0; b < ntiles; b += BLOCK) {
        const long long i = b + threadIdx.x;
        const long long x = i < ntiles ? tile_sum[i] : 0;
        long long tot;
        const long long ex = block_excl_scan(x, &tot);
        if (i < ntiles) tile_sum[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(BLOCK) k_scan_add(long long *out, long long n, const long long *tile_sum) {
    const long long base = (long long)blockIdx.x * SCAN_TILE;
    const long long add = tile_sum[blockIdx.x];
    for (int i = threadIdx.x; i < SCAN_TILE; i += BLOCK)
        if (base + i < n) out[base + i] += add;
}

// ========================================================= frame queue

// Ticket queue of donated frames.  Producers (donating warps) and consumers
// (idle warps) each draw tickets from their own counter with one
// fetch-and-add; ticket t of either side meets at cell t mod cap, whose
// sequence word walks through
//     t  (free for ticket t)  ->  t | CELL_LOCK  (producer t writing)
//        ->  t + 1  (published)  ->  t + cap  (consumed: free for t + cap)
// or, if consumer t leaves before producer t arrives,  t -> t + cap
// (abandoned; producer t then draws another ticket).  A consumer waits on
// its own cell only, so no line is fought over however many warps are idle,
// and every frame reaches exactly one consumer.  Lane 0 only.
constexpr unsigned long long CELL_LOCK = 1ull << 63;

// Producer holding ticket t: locks its cell for writing.  False if consumer t left, or if the
// launch is stopping (the caller keeps its work).  The cell's previous lap ends by itself: its
// frame is being written or goes to a consumer that waits for it.
__device__ bool cell_lock(const SearchCtl &C, unsigned long long t) {
    unsigned long long *seq = C.pseq + t % (unsigned long long)C.pcap;
    for (long long spin = 0;; ++spin) {
        const unsigned long long sv = load_acquire(seq);
        if (sv == t) {
            if (atomicCAS(seq, t, t | CELL_LOCK) == t) return true;
            continue;                                   // consumer t left meanwhile: look again
        }
        if ((sv & ~CELL_LOCK) > t) return false;        // consumer t left
        if ((spin & 63) == 63 && load_relaxed(C.status) != 0) return false;
        if (spin > RESERVE_SPIN_LIMIT) {                // the cell's previous lap never ended
            set_status(C.status, -3);
            return false;
        }
        __nanosleep(128);
    }
}

// Producer: a ticket whose cell is locked for writing, or -1 (the caller keeps its work).
__device__ long long queue_reserve(const SearchCtl &C) {
    for (int a = 0; a < RESERVE_TICKETS && load_relaxed(C.status) == 0; ++a) {
        const unsigned long long t = atomicAdd(C.ptail, 1ull);
        if (cell_lock(C, t)) return (long long)t;
    }
    return -1;
}

// Producer: draws up to `most` consecutive tickets, but only ones that consumers hold already, and
// returns how many (the first one in t).  Consumer tickets only grow in number, so ptail never
// passes phead: however many donors see the same idle warps, together they hand out no more frames
// than there are warps waiting, and no frame lies in a cell that nobody comes for.
__device__ int queue_draw(const SearchCtl &C, int most, unsigned long long &t) {
    unsigned long long tail = load_relaxed(C.ptail);
    for (int a = 0; a < DRAW_TRIES; ++a) {
        const long long waiting = (long long)(load_relaxed(C.phead) - tail);
        if (waiting <= 0) return 0;
        const int n = (int)min((long long)most, waiting);
        const unsigned long long seen = atomicCAS(C.ptail, tail, tail + (unsigned long long)n);
        if (seen == tail) {
            t = tail;
            return n;
        }
        tail = seen;   // another donor was first
    }
    return 0;
}

// Consumer holding ticket t: is its frame published?  (An unordered poll: an acquire at every look
// of every idle warp drops its SM's L1 under the busy ones; acquire_frame fences before it reads.)
__device__ __forceinline__ bool queue_ready(const SearchCtl &C, unsigned long long t) {
    return load_relaxed(C.pseq + t % (unsigned long long)C.pcap) == t + 1;
}

// Consumer holding ticket t wants to leave: true if it left (no frame will
// come to it), false if its frame is published (the caller takes it) or, when
// not stopping, if the cell is still in its previous lap (the caller stays).
// A stopping consumer leaves a cell in its previous lap as it is: a frame
// published there later is found among the unconsumed cells after the launch.
__device__ bool queue_leave(const SearchCtl &C, unsigned long long t, bool stopping) {
    const unsigned long long cap = (unsigned long long)C.pcap;
    unsigned long long *seq = C.pseq + t % cap;
    for (long long spin = 0;; ++spin) {
        const unsigned long long sv = load_acquire(seq);
        if (sv == t + 1) return false;
        if (sv == t) {
            if (atomicCAS(seq, t, t + cap) == t) return true;
            continue;
        }
        if (!(sv & CELL_LOCK) && sv < t) return stopping;   // previous lap still in use
        // locked by a producer, which publishes once its warp has the other cells of its donation
        // (each of them waits for a consumer that is there): wait
        if (spin > RESERVE_SPIN_LIMIT) {
            set_status(C.status, -3);
            return true;
        }
        __nanosleep(128);
    }
}

// Warp-collective: writes frame [j, depth, beg, end, M[0..mlen-1] (+ last)] to the locked cell
// of ticket t and publishes it (`last` >= 0 appends one more image).
__device__ __forceinline__ void publish_frame(const SearchCtl &C, long long t, int j, int depth, int beg, int end,
                                              const int *M, int mlen, int last) {
    const int lane = threadIdx.x & 31;
    int32_t *cell = C.pool + (size_t)(t % C.pcap) * POOL_STRIDE;
    if (lane == 0) { cell[0] = j; cell[1] = depth; cell[2] = beg; cell[3] = end; }
    for (int i = lane; i < mlen; i += 32) cell[FRAME_HDR + i] = M[i];
    if (last >= 0 && lane == 0) cell[FRAME_HDR + mlen] = last;
    __syncwarp();
    if (lane == 0) {
        __threadfence();
        store_release(C.pseq + (t % C.pcap), (unsigned long long)t + 1);   // publish (clears the lock)
        atomicAdd(C.donations, 1ull);
    }
    __syncwarp();
}

// Warp-collective: push one frame.  Returns false if no cell would take it.
__device__ bool push_frame(const SearchCtl &C, int j, int depth, int beg, int end, const int *M, int mlen, int last) {
    long long t = -1;
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(C.outstanding, 1);
        t = queue_reserve(C);
        if (t < 0) atomicSub(C.outstanding, 1);
    }
    t = __shfl_sync(FULL, t, 0);
    if (t < 0) return false;
    publish_frame(C, t, j, depth, beg, end, M, mlen, last);
    return true;
}

// Warp-collective: the same for a warp that is already waiting; false if none is.
__device__ bool push_to_waiting(const SearchCtl &C, int j, int depth, int beg, int end, const int *M, int mlen) {
    long long t = -1;
    if ((threadIdx.x & 31) == 0) {
        unsigned long long at = 0;
        if (queue_draw(C, 1, at) == 1) {
            atomicAdd(C.outstanding, 1);
            if (cell_lock(C, at)) t = (long long)at;
            else atomicSub(C.outstanding, 1);
        }
    }
    t = __shfl_sync(FULL, t, 0);
    if (t < 0) return false;
    publish_frame(C, t, j, depth, beg, end, M, mlen, -1);
    return true;
}

// Warp-collective: push a frame [j, depth, -1, -1, M[0..depth-2], c] for up to `most` lanes of
// `mask` (c: the lane's last image), as many as warps wait, every lane working on its own cell.
// Some cells may not take a frame (a consumer that left): the frames go out lowest lane first, and
// the lanes whose frame was taken, the lowest ones of `mask`, are returned (a checkpoint writes
// what is left of a chunk as one range from its lowest pending survivor on).
__device__ unsigned push_children(const SearchCtl &C, int j, int depth, const int *M, unsigned mask, int most, int c) {
    const int lane = threadIdx.x & 31;
    const unsigned long long cap = (unsigned long long)C.pcap;
    unsigned long long t = 0;
    int n = 0;
    if (lane == 0) {
        n = queue_draw(C, most, t);
        if (n > 0) atomicAdd(C.outstanding, n);   // (this warp's own frame keeps the count above 0)
    }
    n = __shfl_sync(FULL, n, 0);
    if (n == 0) return 0;
    while (__popc(mask) > n) mask &= ~(0x80000000u >> __clz(mask));
    t = __shfl_sync(FULL, t, 0) + __popc(mask & ((1u << lane) - 1u));
    const bool got = ((mask >> lane) & 1u) && cell_lock(C, t);
    __syncwarp();
    const unsigned locked = __ballot_sync(FULL, got);
    int32_t *cell = C.pool + (size_t)(t % cap) * POOL_STRIDE;
    // the r-th locked cell takes the r-th lane's frame
    const int from = got ? (int)__fns(mask, 0, __popc(locked & ((1u << lane) - 1u)) + 1) : lane;
    c = __shfl_sync(FULL, c, from);
    if (got) {
        cell[0] = j; cell[1] = depth; cell[2] = -1; cell[3] = -1;
        cell[FRAME_HDR + depth - 1] = c;
    }
    const unsigned sent = __reduce_or_sync(FULL, got ? 1u << from : 0u);
    for (unsigned m = locked; m; m &= m - 1) {
        int32_t *to = C.pool + (size_t)(__shfl_sync(FULL, t, __ffs(m) - 1) % cap) * POOL_STRIDE + FRAME_HDR;
        for (int i = lane; i < depth - 1; i += 32) to[i] = M[i];
    }
    __syncwarp();
    if (got) {
        __threadfence();
        store_release(C.pseq + (t % cap), t + 1);   // publish (clears the lock)
    }
    if (lane == 0) {
        if (n > __popc(sent)) atomicSub(C.outstanding, n - __popc(sent));
        if (sent) atomicAdd(C.donations, (unsigned long long)__popc(sent));
    }
    __syncwarp();
    return sent;
}

struct Frame {
    int job, depth, beg, end;
    bool counted;   // FRAME_COUNTED: the range's accepted nodes and states are already counted
    bool in_run;    // FRAME_RUN: the range counts in the node's label run
    bool queued;    // it came from another warp
};

// Optional per-warp timing, kept in the warp's own trace record (no registers):
// {start, exit, busy, last frame end, longest frame's duration, its
// job | depth << 16 | origin << 30 (1 frontier, 2 queue), its states, its
// nodes, origin of the current frame, ns spent donating, donation events,
// frames donated, frames taken from the queue, ns and states in them, 0}
// (WTRACE_WORDS words).
struct WarpClock {
    __device__ static unsigned long long *rec(const SearchCtl &C) {
        return C.wtrace + WTRACE_WORDS * ((size_t)blockIdx.x * WARPS_PER_BLOCK + (threadIdx.x >> 5));
    }
    __device__ static void begin(const SearchCtl &C) {
        if (C.wtrace && (threadIdx.x & 31) == 0) rec(C)[0] = globaltimer();
    }
    __device__ static void origin(const SearchCtl &C, int kind) {
        if (C.wtrace && (threadIdx.x & 31) == 0) rec(C)[8] = (unsigned long long)kind;
    }
    __device__ static void frame_in(const SearchCtl &C) {
        if (C.wtrace && (threadIdx.x & 31) == 0) rec(C)[3] = globaltimer();
    }
    __device__ static void frame_out(const SearchCtl &C, const Frame &fr, unsigned long long st,
                                     unsigned long long nd) {
        if (C.wtrace && (threadIdx.x & 31) == 0) {
            unsigned long long *w = rec(C);
            const unsigned long long now = globaltimer(), dur = now - w[3];
            w[2] += dur;
            w[3] = now;   // after the last frame: when the warp last held work
            if (w[8] == 2) { w[12] += 1; w[13] += dur; w[14] += st; }
            if (dur > w[4]) {
                w[4] = dur;
                w[5] = (unsigned long long)fr.job | ((unsigned long long)fr.depth << 16) | (w[8] << 30);
                w[6] = st;
                w[7] = nd;
            }
        }
    }
    __device__ static void finish(const SearchCtl &C) {
        if (C.wtrace && (threadIdx.x & 31) == 0) rec(C)[1] = globaltimer();
    }
    __device__ static unsigned long long don_begin(const SearchCtl &C) {
        return (C.wtrace && (threadIdx.x & 31) == 0) ? globaltimer() : 0ull;
    }
    __device__ static void don_end(const SearchCtl &C, unsigned long long t, int given) {
        if (C.wtrace && (threadIdx.x & 31) == 0) {
            unsigned long long *w = rec(C);
            w[9] += globaltimer() - t;
            w[10] += 1;
            w[11] += (unsigned long long)given;
        }
    }
};


// Warp-collective: append range frame [j, depth (| FRAME_COUNTED), beg, end,
// M[0..depth-1]] to the checkpoint.  Every warp dumps at most two frames per
// level, so a buffer of 2 * kmax frames per warp never overflows.
__device__ void ckpt_push(const SearchCtl &C, int j, int depth, bool counted, int beg, int end, const int *M) {
    const int lane = threadIdx.x & 31;
    unsigned long long slot = 0;
    if (lane == 0) slot = atomicAdd(C.ckpt_n, 1ull);
    slot = __shfl_sync(FULL, slot, 0);
    if ((long long)slot >= C.ckpt_cap) return;
    int32_t *cell = C.ckpt + (size_t)slot * C.ckpt_stride;
    if (lane == 0) { cell[0] = j; cell[1] = depth | (counted ? FRAME_COUNTED : 0); cell[2] = beg; cell[3] = end; }
    for (int i = lane; i < depth; i += 32) cell[FRAME_HDR + i] = M[i];
    __syncwarp();
}

// First index in ascending a[0..n) whose value is >= x (lane 0 searches, all lanes get it).
__device__ int lower_bound_warp(const int32_t *a, int n, int x) {
    int lo = 0;
    if ((threadIdx.x & 31) == 0) {
        int hi = n;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(a + mid) < x) lo = mid + 1; else hi = mid;
        }
    }
    return __shfl_sync(FULL, lo, 0);
}

// Warp-collective: take the next frame (frontier first, then the queue) and
// copy its images into M.  Waits (bounded) while other warps still hold work.
// Returns false when the search is over or stopped.
__device__ bool acquire_frame(const SearchCtl &C, int *M, Frame &fr, unsigned long long deadline) {
    const int lane = threadIdx.x & 31;
    bool idle = false;
    long long spins = 0;
    unsigned backoff = 64;
    unsigned long long idle_since = 0;
    int kind = 0;        // 1 frontier, 2 queue, 0 stop
    long long idx = -1;
    long long ticket = -1;   // consumer ticket held (lane 0)
    for (;;) {
        kind = -1;
        if (lane == 0) {
            if (load_relaxed(C.status) != 0) {
                // stopping: leave the ticket, or take the frame already sent to it
                if (ticket >= 0 && !queue_leave(C, (unsigned long long)ticket, true)) { kind = 2; idx = ticket; }
                else kind = 0;
            } else {
                if (ticket < 0 && load_relaxed(C.fnext) < (unsigned long long)C.nfront) {
                    const unsigned long long f = atomicAdd(C.fnext, 1ull);
                    if ((long long)f < C.nfront) { kind = 1; idx = (long long)f; }
                }
                if (kind < 0) {
                    if (ticket < 0) ticket = (long long)atomicAdd(C.phead, 1ull);
                    if (queue_ready(C, (unsigned long long)ticket)) { kind = 2; idx = ticket; }
                }
                // all work done: no frame can come to the ticket any more
                if (kind < 0 && load_relaxed(C.outstanding) == 0) kind = 0;
            }
            if (kind < 0) {
                if (!idle) { atomicAdd(C.idle, 1); idle = true; idle_since = globaltimer(); }
                // optional early exit of a warp that found no work for a while (it leaves its
                // ticket first; a frame already sent to it is taken instead), so the freed block
                // slots serve kernels launched on other streams
                else if (C.idle_exit_ns != 0 && globaltimer() - idle_since > C.idle_exit_ns) {
                    if (queue_leave(C, (unsigned long long)ticket, false)) kind = 0;
                    else if (queue_ready(C, (unsigned long long)ticket)) { kind = 2; idx = ticket; }
                    else idle_since = globaltimer();   // previous lap still in use: stay a while
                }
                if (kind < 0 && (++spins & 1023) == 0) {
                    // the stop paths set the status; the next round leaves the ticket.  A warp idle
                    // far longer than any search leaves a frame to wait ends the launch with an error.
                    const unsigned long long now = globaltimer();
                    if ((C.cancel != nullptr && *C.cancel != 0)) set_status(C.status, -6);
                    else if (deadline != 0 && now > deadline) set_status(C.status, -5);
                    else if (now - idle_since > IDLE_GUARD_NS) set_status(C.status, -3);
                }
            }
        }
        kind = __shfl_sync(FULL, kind, 0);
        if (kind >= 0) break;
        // exponential backoff: one warp per block polls often, the others rarely
        __nanosleep(backoff);
        if (backoff < ((threadIdx.x >> 5) == 0 ? IDLE_BACKOFF_FAST : IDLE_BACKOFF_SLOW)) backoff <<= 1;
    }
    if (lane == 0 && idle) atomicSub(C.idle, 1);
    if (kind == 0) return false;
    WarpClock::origin(C, kind);
    idx = __shfl_sync(FULL, idx, 0);
    const int32_t *src;
    if (kind == 1) {
        const long long g = idx * (long long)C.shard_count + C.shard_index;
        src = C.front_ptr ? C.front_ptr[g] : C.front + g * C.fstride;
    } else {
        if (lane == 0) __threadfence();
        __syncwarp();
        src = C.pool + (size_t)(idx % C.pcap) * POOL_STRIDE;
    }
    const int dw = src[1];
    fr.job = src[0]; fr.depth = dw & FRAME_DEPTH_MASK; fr.counted = (dw & FRAME_COUNTED) != 0;
    fr.in_run = (dw & FRAME_RUN) != 0;
    fr.queued = kind == 2;
    fr.beg = src[2]; fr.end = src[3];
    for (int i = lane; i < fr.depth; i += 32) M[i] = src[FRAME_HDR + i];
    __syncwarp();
    if (kind == 2 && lane == 0) {
        __threadfence();
        store_release(C.pseq + (idx % C.pcap), (unsigned long long)idx + C.pcap);
    }
    return true;
}

// Periodic checks by lane 0: cancellation, deadline, budget, other warps'
// errors.  Returns nonzero (warp-uniform) when the warp must stop.
__device__ __forceinline__ int must_stop(const SearchCtl &C, const JobDesc &J, unsigned long long local_states,
                                         unsigned long long deadline, unsigned long long now,
                                         unsigned long long &last_cancel) {
    int stop = 0;
    if ((threadIdx.x & 31) == 0) {
        const bool read_cancel = C.cancel != nullptr && now - last_cancel >= CANCEL_CHECK_NS;
        if (read_cancel) last_cancel = now;
        if (load_relaxed(C.status) != 0) stop = 1;
        else if (read_cancel && *C.cancel != 0) { set_status(C.status, -6); stop = 1; }
        else if (deadline != 0 && globaltimer() > deadline) { set_status(C.status, -5); stop = 1; }
        else if (C.budget > 0 && (long long)(*(volatile unsigned long long *)(J.ctr + 1) + local_states) > C.budget) {
            set_status(C.status, -4); stop = 1;
        }
    }
    return __shfl_sync(FULL, stop, 0);
}

// Warp-uniform: has CHECK_NS of device time passed since the last check?
__device__ __forceinline__ bool time_to_check(unsigned long long &last) {
    unsigned long long now = 0;
    if ((threadIdx.x & 31) == 0) now = globaltimer();
    now = __shfl_sync(FULL, now, 0);
    if (now - last < CHECK_NS) return false;
    last = now;
    return true;
}

// Warp-uniform: should this warp donate now?  Donation is wanted while more
// warps are idle than frames wait in the queue; a donor first takes one of
// those (idle - queued) slots, so a few donors, not every busy warp, answer
// one idle warp.  A true result must be paired with donation_done().
__device__ __forceinline__ bool donation_claim(const SearchCtl &C) {
    int ok = 0;
    if ((threadIdx.x & 31) == 0 && C.donate) {
        // consumer tickets not yet matched by a producer = idle warps waiting for a frame
        const long long waiting = (long long)(load_relaxed(C.phead) - load_relaxed(C.ptail));
        if (waiting > 0 && atomicAdd(C.promised, 1) < waiting) ok = 1;
        else if (waiting > 0) atomicSub(C.promised, 1);
    }
    return __shfl_sync(FULL, ok, 0) != 0;
}

__device__ __forceinline__ void donation_done(const SearchCtl &C) {
    if ((threadIdx.x & 31) == 0) atomicSub(C.promised, 1);
    __syncwarp();
}

// ===================================================== search: CSR kernel
//
// One warp owns one depth-first search.  A level's candidates are its shortest
// label run, on targets without runs the row of M(P(mu_i)) (or V_t / D(mu_i)
// when mu_i is unparented), scanned 32 at a time, one candidate per lane; each
// lane makes its candidate's local tests, the constraints are tested spread over
// the warp (cand_chunk), and a ballot compacts the chunk's survivors.  Per warp,
// shared memory holds M and the level records; the job's pointers stay in registers.

__host__ __device__ __forceinline__ size_t round16(size_t x) { return (x + 15) & ~(size_t)15; }

// What a level's candidates are entries of.
enum : int16_t { LIST_VERTICES = 0, LIST_DOMAIN, LIST_ROW, LIST_IN_ROW, LIST_RUN, LIST_IN_RUN };

struct LvCsr {
    int base;                // offset of the level's candidate list in its array
    int cur, end;            // unscanned candidates [cur, end)
    unsigned mask;           // survivors of the last scanned chunk, not yet descended
    int cbase;               // index of that chunk's first candidate
    int raw;                 // the node's raw candidate count (its states)
    int len;                 // length of the list
    int16_t kind, skip;      // LIST_*, and the constraint the list itself satisfies
};

__host__ __device__ __forceinline__ size_t csr_smem_per_warp(int kmax) {
    return round16((size_t)kmax * sizeof(LvCsr) + ((size_t)kmax + 32) * sizeof(int));
}

// A job's pointers in registers, read like JobRef.
struct CsrJob {
    const int32_t *rowptr_, *col_, *elab_, *irowptr_, *icol_, *ielab_, *indeg_, *ulist_, *hub_slot_, *plidx_;
    const int2 *vld_;
    const uint64_t *filt_, *adj_, *hub_bits_;
    const BackEdge *back_;
    const PosInfo *pos;
    const LabelRuns *runs_;
    int n_, dw_, k, flags_;
    __device__ __forceinline__ const int32_t *rowptr() const { return rowptr_; }
    __device__ __forceinline__ const int32_t *col() const { return col_; }
    __device__ __forceinline__ const int32_t *elab() const { return elab_; }
    __device__ __forceinline__ const int32_t *irowptr() const { return irowptr_; }
    __device__ __forceinline__ const int32_t *icol() const { return icol_; }
    __device__ __forceinline__ const int32_t *ielab() const { return ielab_; }
    __device__ __forceinline__ const int32_t *indeg() const { return indeg_; }
    __device__ __forceinline__ const int32_t *hub_slot() const { return hub_slot_; }
    __device__ __forceinline__ const uint64_t *hub_bits() const { return hub_bits_; }
    __device__ __forceinline__ const uint64_t *adj() const { return adj_; }
    __device__ __forceinline__ const int2 *vld() const { return vld_; }
    __device__ __forceinline__ const LabelRuns *runs() const { return runs_; }
    __device__ __forceinline__ const uint64_t *filt() const { return filt_; }
    __device__ __forceinline__ const BackEdge *back() const { return back_; }
    __device__ __forceinline__ const int32_t *ulist() const { return ulist_; }
    __device__ __forceinline__ const int32_t *plidx() const { return plidx_; }
    __device__ __forceinline__ int n() const { return n_; }
    __device__ __forceinline__ int dw() const { return dw_; }
    __device__ __forceinline__ int flags() const { return flags_; }
};

// A level's list as cand_chunk reads it.
template <bool DIR>
__device__ __forceinline__ Cand csr_list(const CsrJob &B, const PosV &p, const LvCsr &L, const int *M) {
    Cand S;
    S.base = L.base;
    S.len = L.len;
    S.raw = L.raw;
    S.skip = L.skip;
    S.next = -1;
    S.elab = nullptr;
    S.li = -1;
    S.lab = p.pel;
    switch (L.kind) {
        case LIST_VERTICES: S.ids = nullptr; break;
        case LIST_DOMAIN: S.ids = B.ulist_; break;
        case LIST_ROW: S.ids = B.col_; S.elab = B.elab_; break;
        case LIST_IN_ROW: S.ids = B.icol_; S.elab = B.ielab_; break;
        default:
            S.ids = reinterpret_cast<const int32_t *>(DIR && L.kind == LIST_IN_RUN ? B.runs_->icol : B.runs_->col);
            S.elab = DIR && L.kind == LIST_IN_RUN ? B.runs_->ielab : B.runs_->elab;
            S.li = B.plidx_[p.pv];
            if (L.skip > 0 && (B.flags_ & JOB_ELAB)) S.lab = constraint<DIR>(B, p, L.skip, M).lab;
    }
    return S;
}

template <bool DIR>
__global__ void __launch_bounds__(BLOCK, 3) k_search_csr(const JobDesc *jobs, SearchCtl C, int kmax) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char *base = smem + wib * csr_smem_per_warp(kmax);
    LvCsr *lv = reinterpret_cast<LvCsr *>(base);
    int *M = reinterpret_cast<int *>(lv + kmax);
    int *Cs = M + kmax;

    const unsigned long long deadline = C.deadline_ns ? globaltimer() + C.deadline_ns : 0ull;
    Frame fr;
    unsigned iter = 0, last_don_iter = 0;
    unsigned long long last_check = 0, last_don_ns = 0, last_cancel = 0;
    int cur_job = -1;
    CsrJob B;
    WarpClock::begin(C);
    if (threadIdx.x == 0) atomicMax(C.span, ~globaltimer());
    while (acquire_frame(C, M, fr, deadline)) {
        WarpClock::frame_in(C);
        const JobDesc &J = jobs[fr.job];
        if (fr.job != cur_job) {
            cur_job = fr.job;
            B.rowptr_ = J.t.rowptr; B.col_ = J.t.col; B.elab_ = J.t.elab;
            B.irowptr_ = J.t.irowptr; B.icol_ = J.t.icol; B.ielab_ = J.t.ielab; B.indeg_ = J.t.indeg;
            B.ulist_ = J.ulist; B.vld_ = J.t.vld; B.filt_ = J.filt; B.adj_ = J.t.adj; B.back_ = J.back; B.pos = J.pos;
            B.hub_slot_ = J.t.hub_slot; B.hub_bits_ = J.t.hub_bits; B.runs_ = J.t.runs; B.plidx_ = J.plidx;
            B.n_ = J.t.n; B.dw_ = J.t.dw; B.k = J.k; B.flags_ = J.flags;
        }
        const int k = B.k, d0 = fr.depth;
        // a counted frame re-tests its range at level d0 without counting it again
        const int quiet = fr.counted ? d0 : -1;
        unsigned long long st = 0, nd = 0, mt = 0, hs = 0;   // the frame's totals
        // since the last fold (every 64 iterations): an iteration adds at most 32 nodes and a
        // candidate list below 2^24 states (longer lists go straight to the 64-bit total)
        unsigned st32 = 0, nd32 = 0, mt32 = 0;
        bool counts0 = true;   // the frame counted its first node's states
        // a frame of the frontier (or a part of one) that starts on the last level but one has nothing
        // shallower to give: halves of its range, if that is long, have one level below them (a path of
        // 3 on a 100,000-vertex network of 2 labels, from depth 1: 25 ms on one hub's frame -> 3.6)
        const bool last_but_one = d0 + 2 == k && (!fr.queued || fr.beg >= 0);
        // scan the next 32 candidates [cur, ..) of level `l`'s list
        auto scan = [&](int l, const PosV &p, const Cand &S, int cur, int end) {
            int c;
            unsigned bal = cand_chunk<DIR>(B, p, B.pos + l, S, cur, end, M, Cs, c);
            if (l != quiet) nd32 += __popc(bal);
            if (l == k - 1) {
                mt32 += __popc(bal);
                if (bal) {
                    // hash prefix sum_{t < l} g(mu_t, M_t), only when this chunk has matches
                    unsigned long long ps = 0;
                    for (int t = lane; t < l; t += 32) ps += gterm(__ldg(&B.pos[t].pv), M[t]);
                    ps = warp_sum(ps);
                    if ((bal >> lane) & 1u) {
                        hs += fmix64(ps + gterm(p.pv, c));
                        if (J.mbuf) emit_match(J, M, l, c);
                    }
                }
                bal = 0;
            }
            __syncwarp();
            if (lane == 0) { lv[l].cur = min(cur + 32, end); lv[l].mask = bal; lv[l].cbase = cur; }
            __syncwarp();
            return bal != 0 || end - cur > 32;   // something is left on the level
        };
        // set up level `l` (positions 0..l-1 assigned), count the node's states -- a range
        // frame counts them if it starts the node, a counted frame not at all -- and, below the
        // frame's first node, scan its first candidates while the list is at hand.  Returns
        // whether anything is left on the level: most nodes at the bottom have one chunk, and a
        // round of the loop to find them done cost as much as some of them.
        auto setup = [&](int l, int beg, int endv, bool in_run) {
            const PosV p = load_pos(B.pos + l);
            const Cand S = pick_warp<DIR>(B, p, B.pos + l, M);
            int cur, end;
            const bool counts = list_range<DIR>(B, p, S, M, beg, endv, in_run, cur, end);
            int kind = p.par < 0 ? (S.ids ? LIST_DOMAIN : LIST_VERTICES) : LIST_ROW;
            if (p.par >= 0) {
                if (B.runs_ != nullptr)
                    kind = DIR && S.ids == reinterpret_cast<const int32_t *>(B.runs_->icol) ? LIST_IN_RUN : LIST_RUN;
                else if (DIR && (p.flags & POS_IN_ROW)) kind = LIST_IN_ROW;
            }
            __syncwarp();
            if (lane == 0) {
                lv[l].base = S.base; lv[l].cur = cur; lv[l].end = end; lv[l].mask = 0; lv[l].cbase = 0;
                lv[l].raw = S.raw; lv[l].len = S.len; lv[l].kind = (int16_t)kind; lv[l].skip = (int16_t)S.skip;
            }
            __syncwarp();
            if (l == d0) counts0 = counts;
            if (counts && l != quiet) {
                if (S.raw < (1 << 24)) st32 += (unsigned)S.raw;
                else st += (unsigned long long)S.raw;
            }
            if (l > d0 && cur < end) return scan(l, p, S, cur, end);
            return cur < end;
        };
        // candidate of entry e of level l's list
        auto entry = [&](const LvCsr &L, int e) {
            if (L.kind >= LIST_RUN) return __ldg(&(DIR && L.kind == LIST_IN_RUN ? B.runs_->icol : B.runs_->col)[L.base + e]).x;
            const int32_t *ids = L.kind == LIST_VERTICES ? nullptr
                                 : L.kind == LIST_DOMAIN ? B.ulist_
                                 : L.kind == LIST_ROW    ? B.col_ : B.icol_;
            return ids ? __ldg(ids + L.base + e) : L.base + e;
        };
        setup(d0, fr.beg, fr.end, fr.in_run);
        int lvl = d0;
        bool stopped = false;
        for (;;) {
            if (((++iter) & 63) == 0) {
                st += st32; nd += nd32; mt += mt32;
                st32 = nd32 = mt32 = 0;
            }
            if ((iter & 7) == 0 && time_to_check(last_check)) {
                if (C.budget > 0) {
                    st += st32;
                    st32 = 0;
                    if (lane == 0) atomicAdd(J.ctr + 1, st);
                    st = 0;
                }
                if (must_stop(C, J, st, deadline, last_check, last_cancel)) { stopped = true; break; }
            }
            if (C.donate && (iter - last_don_iter >= (unsigned)C.donate_iters ||
                             ((iter & 7) == 0 && last_check - last_don_ns >= C.donate_ns))) {
                // idle warps waiting for a frame (their tickets run ahead of the producers')?
                last_don_iter = iter;
                last_don_ns = last_check;
                int want = 0;
                if (lane == 0)
                    want = (int)max(-1ll, min(32ll, (long long)(load_relaxed(C.phead) - load_relaxed(C.ptail))));
                want = __shfl_sync(FULL, want, 0);
                // donate the shallowest unexplored work: half of an unscanned range, else up to
                // `gran` pending survivors as new search nodes
                const int levels = last_but_one ? 1 : DONATE_MIN_LEVELS;
                for (int l = d0; want > 0 && l <= lvl && l + 1 + levels <= k; ++l) {
                    LvCsr &L = lv[l];
                    int rem = L.end - L.cur;
                    if (rem >= 64 && L.kind >= LIST_RUN) {   // past the entries no part may start in
                        const PosV p = load_pos(B.pos + l);
                        const int drop = run_drop<DIR>(B, p, csr_list<DIR>(B, p, L, M), M);
                        __syncwarp();
                        if (lane == 0 && L.cur < drop) L.cur = min(drop, L.end);
                        __syncwarp();
                        rem = L.end - L.cur;
                    }
                    if (rem >= 64) {
                        const int mid = L.cur + ((rem / 2 + 31) & ~31);
                        const int run = L.kind >= LIST_RUN ? FRAME_RUN : 0;
                        if (push_to_waiting(C, fr.job, l | (l == quiet ? FRAME_COUNTED : 0) | run, mid, L.end, M, l)) {
                            __syncwarp();
                            if (lane == 0) L.end = mid;
                            __syncwarp();
                        }
                        break;
                    }
                    if (last_but_one) break;   // (no single nodes)
                    const unsigned m = L.mask;
                    // (the current level keeps one for this warp, which would else be out of work)
                    const int most = min(min(want, C.gran), __popc(m) - (l == lvl ? 1 : 0));
                    if (most > 0) {
                        // the lowest ones, one per lane
                        const int c = (m >> lane) & 1u ? entry(L, L.cbase + lane) : 0;
                        const unsigned sent = push_children(C, fr.job, l + 1, M, m, most, c);
                        if (lane == 0) L.mask &= ~sent;
                        __syncwarp();
                        break;
                    }
                }
            }
            LvCsr &L = lv[lvl];
            const unsigned mask = L.mask;
            if (mask == 0) {
                const int cur = L.cur, end = L.end;
                if (cur >= end) {
                    if (lvl == d0) break;
                    --lvl;
                    continue;
                }
                const PosV p = load_pos(B.pos + lvl);
                scan(lvl, p, csr_list<DIR>(B, p, L, M), cur, end);
                continue;
            }
            // descend into the lowest pending survivor
            const int c = entry(L, L.cbase + __ffs(mask) - 1);
            __syncwarp();
            if (lane == 0) {
                L.mask = mask & (mask - 1);
                M[lvl] = c;
            }
            __syncwarp();
            if (setup(lvl + 1, -1, 0, false)) ++lvl;
        }
        if (stopped && C.ckpt != nullptr) {
            // checkpoint, per level: the part of the current chunk from its lowest pending
            // survivor on (already counted; survivors are taken lowest first), then the
            // unscanned rest of the range (counted only if the frame itself was); both as ranges
            // of the parent's row.  A part left from entry 0 on counts the node's states again
            // when it is resumed: they are taken back here.
            for (int l = d0; l <= lvl; ++l) {
                const LvCsr L = lv[l];
                const PosV p = load_pos(B.pos + l);
                const Cand S = csr_list<DIR>(B, p, L, M);
                const int cb = L.mask ? L.cbase + __ffs(L.mask) - 1 : L.cur;
                int beg, end;
                if (l == quiet) {
                    if (cb < L.end) {
                        row_range<DIR>(B, p, S, M, cb, L.end, beg, end);
                        ckpt_push(C, fr.job, l, true, beg, end, M);
                    }
                } else {
                    if (cb < L.cur) {
                        row_range<DIR>(B, p, S, M, cb, L.cur, beg, end);
                        ckpt_push(C, fr.job, l, true, beg, end, M);
                    }
                    const int cur = L.cur < L.end && S.li >= 0 ? max(L.cur, run_drop<DIR>(B, p, S, M)) : L.cur;
                    if (cur < L.end) {
                        row_range<DIR>(B, p, S, M, cur, L.end, beg, end);
                        const bool counted = l > d0 || counts0;
                        if (counted && L.cur == 0) beg = 0;   // scan not begun: the whole node
                        if (counted && beg == 0) st -= (unsigned long long)L.raw;
                        ckpt_push(C, fr.job, l, false, beg, end, M);
                    }
                }
            }
        }
        st += st32; nd += nd32; mt += mt32;
        hs = warp_sum(hs);
        if (lane == 0) {
            atomicAdd(J.ctr + 0, mt);
            atomicAdd(J.ctr + 1, st);
            atomicAdd(J.ctr + 2, nd);
            atomicAdd(J.ctr + 3, hs);
            if (!stopped) atomicSub(C.outstanding, 1);
        }
        __syncwarp();
        WarpClock::frame_out(C, fr, st, nd);
        if (stopped) break;
    }
    WarpClock::finish(C);
    if ((threadIdx.x & 31) == 0) atomicMax(C.span + 1, globaltimer());
}

// One warp per checkpoint frame: a label-run range becomes the same part of the parent's row.
template <bool DIR>
__global__ void __launch_bounds__(BLOCK) k_frames_to_rows(const JobDesc *jobs, int32_t *frames, long long n,
                                                          long long pitch, const unsigned long long *seq) {
    const long long f = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (f >= n) return;
    if (seq != nullptr) {   // a queue cell that is not published holds no frame
        const unsigned long long sv = seq[f];
        if (sv == 0 || (sv & CELL_LOCK) || (sv - 1) % (unsigned long long)n != (unsigned long long)f) return;
    }
    int32_t *fr = frames + f * pitch;
    const int dw = fr[1];
    if (!(dw & FRAME_RUN)) return;
    const JobDesc &J = jobs[fr[0]];
    const JobRef v{&J};
    const PosInfo *P = J.pos + (dw & FRAME_DEPTH_MASK);
    const PosV p = load_pos(P);
    const int *M = fr + FRAME_HDR;
    const Cand S = pick_warp<DIR>(v, p, P, M);
    int lo, hi, beg = 1, end = 1;   // (an empty part)
    const bool counts = list_range<DIR>(v, p, S, M, fr[2], fr[3], true, lo, hi);
    if (lo < hi) row_range<DIR>(v, p, S, M, lo, hi, beg, end);
    if (counts) {
        end = lo < hi ? end : 0;
        beg = 0;
    }
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        fr[1] = dw & ~FRAME_RUN;
        fr[2] = beg;
        fr[3] = end;
    }
}

// ================================================== search: bitset kernel
//
// Candidate set of position i as one AND over bitset rows (dense targets):
//   S_i = D(mu_i) & A[M(P(mu_i))] & AND_j A[M(mu_j)] & ~used
// where D is the domain (RI-DS) or the label/degree filter (RI), A the
// adjacency bitset and `used` the images M_0..M_{i-1} (rule 1).  Lane l owns
// words l, l + 32, ... (NWL per lane, 1 to 4, as few as the row needs: every word per lane is an
// AND and a popcount in each expansion; 79 words on 3 instead of 4, four patterns on a
// 5,003-vertex target: 12.1 -> 11.0 ms, another four 20.3 -> 18.7).
//
// Per warp, registers hold the used-vertex bitset (lane l: words l + 32 w) and
// shared memory holds M, a compact copy of the job's position table, and for
// every level a list of up to BitsLayout<KM>::LCAP pending survivors; a level with
// more survivors keeps its
// bitset in the warp's slab of global scratch (`SearchCtl::slab`) instead.

// Capacity of a level's survivor list in shared memory: 64 for patterns of up
// to 32 vertices (measured fastest on the dense workload), 16 beyond so that
// four blocks of eight warps still fit an SM.  (The length byte reserves 0xff.)
constexpr uint8_t LIST_SPILLED = 0xff;

// Pattern-size class of a bitset-kernel launch: its per-warp shared layout is
// fixed at compile time for patterns of at most KM vertices.
// (A smaller class keeps shared memory, and so the L1 left beside it for the adjacency rows,
// no larger than the patterns need: 24 vertices take 31 KB per block, 32 take 42 KB.)
__host__ __device__ constexpr int bits_km(int kmax) {
    return kmax <= 24 ? 24 : (kmax <= 32 ? 32 : (kmax <= 64 ? 64 : KMAX));
}

struct __align__(16) PosB {
    int16_t pv, par, bb, bc;  // pattern vertex, parent position, back edges [bb, bb + bc) other than
                              // one to position i - 1 (that one, if any, is stored right after them)
    int32_t ucnt;             // raw candidates of an unparented position
    int32_t abf;              // algorithmic bytes of one expansion (rows ANDed x dw x 8, low 28 bits),
                              // flags PREV_ADJ / PREV_PAR above them
};
constexpr int32_t PREV_ADJ = 1 << 28;   // mu_{i-1} is adjacent to mu_i (as parent or back edge)
constexpr int32_t PREV_PAR = 1 << 29;   // ... and is its parent
constexpr int32_t ABYTES_MASK = (1 << 28) - 1;

// Per-warp shared memory of the bitset kernel, at offsets fixed by KM: the
// position table (16-byte records), the frame's range (for checkpoints), M,
// the survivor lists and their lengths, and the back-edge positions.
template <int KM>
struct BitsLayout {
    static constexpr int LCAP = KM <= 32 ? 64 : 16;   // (KM 24 and 32: 64 entries)
    static constexpr size_t TAB = 0;
    static constexpr size_t FRANGE = TAB + (size_t)KM * 16;
    static constexpr size_t MOFF = FRANGE + 8;
    static constexpr size_t LST = MOFF + (size_t)KM * 4;
    static constexpr size_t LCNT = LST + (size_t)KM * LCAP * 2;
    static constexpr size_t TBACK = LCNT + (size_t)KM;
    static constexpr size_t BYTES = (TBACK + (size_t)KM * (KM - 1) / 2 + 16 + 15) & ~(size_t)15;
};

__host__ __device__ __forceinline__ size_t bits_smem_per_warp(int kmax, int nwl) {
    switch (bits_km(kmax)) {
        case 24: return BitsLayout<24>::BYTES;
        case 32: return BitsLayout<32>::BYTES;
        case 64: return BitsLayout<64>::BYTES;
        default: return BitsLayout<KMAX>::BYTES;
    }
}

__host__ __device__ __forceinline__ size_t bits_slab_words_per_warp(int kmax, int nwl) {
    return (size_t)bits_km(kmax) * nwl * 32;
}

struct BitsJob {
    const uint64_t *filt, *adj;
    const int2 *vld;
    int dw, k;
};

// One warp's state: its shared-memory block (offsets from BitsLayout<KM>) and
// its slab of global scratch (level bitsets of more survivors than a list holds).
template <int KM>
struct BitsWarp {
    using L = BitsLayout<KM>;
    static constexpr int LCAP = L::LCAP;
    unsigned char *base;
    uint64_t *slab;    // global: [KM][NWL * 32]
    // Level l's list length (LIST_SPILLED: its survivors are a slab bitset).  Patterns of up
    // to 32 vertices keep the lengths in a register, lane l holding level l's, so a pop
    // reads it with one shuffle and writes it with one select, no shared-memory store or
    // warp sync; larger ones keep them in shared memory.
    int lcr;
    __device__ __forceinline__ int lc(int l) const {
        if constexpr (KM <= 32) return __shfl_sync(FULL, lcr, l);
        else return lcnt()[l];
    }
    __device__ __forceinline__ void set_lc(int l, int v) {
        if constexpr (KM <= 32) {
            lcr = (threadIdx.x & 31) == l ? v : lcr;
        } else {
            __syncwarp();
            if ((threadIdx.x & 31) == 0) lcnt()[l] = (uint8_t)v;
            __syncwarp();
        }
    }
    __device__ __forceinline__ PosB *tab() const { return reinterpret_cast<PosB *>(base + L::TAB); }
    __device__ __forceinline__ int *frange() const { return reinterpret_cast<int *>(base + L::FRANGE); }
    __device__ __forceinline__ int *M() const { return reinterpret_cast<int *>(base + L::MOFF); }
    __device__ __forceinline__ uint16_t *lst() const { return reinterpret_cast<uint16_t *>(base + L::LST); }
    __device__ __forceinline__ uint8_t *lcnt() const { return base + L::LCNT; }
    __device__ __forceinline__ uint8_t *tback() const { return base + L::TBACK; }
};

template <int NWL>
__device__ __forceinline__ void used_flip(uint64_t (&used)[NWL], int v) {
    // lane (q mod 32) holds word q of the used bitset in register used[q / 32]
    const int q = v >> 6;
    if ((threadIdx.x & 31) == (q & 31)) {
        const uint64_t bit = 1ull << (v & 63);
        if (NWL == 1) {
            used[0] ^= bit;   // v < 64 * 32: q < 32
        } else {
#pragma unroll
            for (int w = 0; w < NWL; ++w)
                if (w == (q >> 5)) used[w] ^= bit;
        }
    }
}

// This lane's words of row x of the adjacency bitset, ANDed into s.
template <int NWL>
__device__ __forceinline__ void and_row(const uint64_t *adj, int dw, int x, uint64_t (&s)[NWL]) {
    const uint64_t *X = adj + (size_t)x * dw;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int w = 0; w < NWL; ++w) {
        const int q = lane + 32 * w;
        if (q < dw) s[w] &= __ldg(X + q);
    }
}

// The part of position i's candidate set that does not depend on M[i-1]:
//   P_i = D(mu_i) & A[M(P(mu_i))] (unless the parent is position i - 1)
//         & AND over the other back-neighbours j < i - 1 of A[M_j] & ~used
// (`used` = images of positions 0..i-2).  With `with_prev` the rows of
// position i - 1 are ANDed too (then `used` must hold M_{i-1} as well), which
// gives the whole candidate set S_i.  `len` receives the raw candidate count
// when it does not depend on M[i-1] (else 0).
template <int NWL, int KM>
__device__ __forceinline__ void bits_rows(const BitsJob &B, const BitsWarp<KM> &W, const PosB &p, int i, bool with_prev,
                                          const uint64_t (&used)[NWL], uint64_t (&s)[NWL], int &len) {
    const int lane = threadIdx.x & 31;
    const int dw = B.dw;
    const uint64_t *F = B.filt + (size_t)p.pv * dw;
    const int *M = W.M();
#pragma unroll
    for (int w = 0; w < NWL; ++w) {
        const int q = lane + 32 * w;
        s[w] = q < dw ? F[q] : 0ull;
    }
    len = p.ucnt;
    if (p.par >= 0) {
        if (with_prev || !(p.abf & PREV_PAR)) {
            const int a = M[p.par];
            and_row<NWL>(B.adj, dw, a, s);
            len = __ldg(B.vld + a).y;
        } else {
            len = 0;
        }
    }
#pragma unroll 2
    for (int b = 0; b < p.bc; ++b) and_row<NWL>(B.adj, dw, M[W.tback()[p.bb + b]], s);
    if (with_prev && (p.abf & PREV_ADJ) && !(p.abf & PREV_PAR)) and_row<NWL>(B.adj, dw, M[i - 1], s);
#pragma unroll
    for (int w = 0; w < NWL; ++w) s[w] &= ~used[w];
}

// Count the survivors of position i's candidate set s (the accepted nodes) and
// either hash them as matches (leaf) or keep them as level i's pending
// survivors: a short list in shared memory, else the bitset in the slab.
// With none, level i's list is left as it was: the caller does not descend.
// `st` and `ab` are 32-bit: one expansion adds at most n_t <= 8192 states and
// (k_max + 1) x 128 x 8 bytes, and the caller folds them into 64-bit totals
// every 64 expansions.  M[0..i-1] must be in shared memory when the set has
// matches (the hash and the match rows read them).
template <int NWL, int KM, bool RANGE = false>
__device__ __forceinline__ int bits_finish(const JobDesc &J, BitsWarp<KM> &W, uint64_t (&s)[NWL], int i, int pv,
                                           bool leaf, unsigned long long &hs, int vlo = 0, int vhi = 0x7fffffff) {
    const int lane = threadIdx.x & 31;
    int cnt = 0;
#pragma unroll
    for (int w = 0; w < NWL; ++w) {
        if (RANGE) {
            // a range frame: keep the candidates with vertex ids in [vlo, vhi]
            const int b0 = (lane + 32 * w) * 64;
            if (vhi < b0 || vlo > b0 + 63) {
                s[w] = 0;
            } else {
                const int lo = vlo > b0 ? vlo - b0 : 0, hi = vhi < b0 + 63 ? vhi - b0 : 63;
                s[w] &= (~0ull << lo) & (~0ull >> (63 - hi));
            }
        }
        cnt += __popcll(s[w]);
    }
    const int total = __reduce_add_sync(FULL, (unsigned)cnt);
    if (total == 0) return 0;
    if (leaf) {
        // hash prefix sum_{t < i} g(mu_t, M_t), computed only when matches exist
        const int *M = W.M();
        unsigned long long ps = 0;
        for (int t = lane; t < i; t += 32) ps += gterm(W.tab()[t].pv, M[t]);
        ps = warp_sum(ps);
#pragma unroll
        for (int w = 0; w < NWL; ++w) {
            const int q = lane + 32 * w;
            uint64_t y = s[w];
            while (y) {
                const int bit = __ffsll((long long)y) - 1;
                const int vtx = q * 64 + bit;
                hs += fmix64(ps + gterm(pv, vtx));
                if (J.mbuf) emit_match(J, M, i, vtx);
                y &= y - 1;
            }
        }
        return total;
    }
    if (total <= W.LCAP) {
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        uint16_t *L = W.lst() + i * W.LCAP;
        int o = incl - cnt;
#pragma unroll
        for (int w = 0; w < NWL; ++w) {
            const int q = lane + 32 * w;
            uint64_t y = s[w];
            while (y) {
                L[o++] = (uint16_t)(q * 64 + __ffsll((long long)y) - 1);
                y &= y - 1;
            }
        }
        __syncwarp();
        W.set_lc(i, total);
    } else {
        uint64_t *Sl = W.slab + (size_t)i * NWL * 32;
#pragma unroll
        for (int w = 0; w < NWL; ++w) Sl[w * 32 + lane] = s[w];
        __syncwarp();
        W.set_lc(i, LIST_SPILLED);
    }
    return total;
}

// Next pending survivor of level l (warp-uniform, -1 if none); removes it.
template <int NWL, int KM>
__device__ __forceinline__ int bits_next(BitsWarp<KM> &W, int l) {
    const int lane = threadIdx.x & 31;
    const int c = W.lc(l);
    if (c != LIST_SPILLED) {
        if (c == 0) return -1;
        const int v = W.lst()[l * W.LCAP + c - 1];
        W.set_lc(l, c - 1);
        return v;
    }
    uint64_t *S = W.slab + (size_t)l * NWL * 32;
#pragma unroll
    for (int w = 0; w < NWL; ++w) {
        const uint64_t m = S[w * 32 + lane];
        const unsigned bal = __ballot_sync(FULL, m != 0);
        if (bal) {
            const int L = __ffs(bal) - 1;
            const uint64_t mw = __shfl_sync(FULL, m, L);
            const int bit = __ffsll((long long)mw) - 1;
            __syncwarp();
            if (lane == L) S[w * 32 + lane] = mw & (mw - 1);
            __syncwarp();
            return ((L + 32 * w) << 6) + bit;
        }
    }
    return -1;
}

// Put a survivor back at level l (the donation queue was full).
template <int NWL, int KM>
__device__ __forceinline__ void bits_unnext(BitsWarp<KM> &W, int l, int v) {
    const int lane = threadIdx.x & 31;
    const int c = W.lc(l);
    __syncwarp();
    if (c != LIST_SPILLED) {
        if (lane == 0) W.lst()[l * W.LCAP + c] = (uint16_t)v;
        __syncwarp();
        W.set_lc(l, c + 1);
    } else {
        const int q = v >> 6;
        if (lane == (q & 31)) W.slab[(size_t)l * NWL * 32 + (q >> 5) * 32 + lane] |= 1ull << (v & 63);
        __syncwarp();
    }
}

template <int NWL, int KM>
__global__ void __launch_bounds__(BLOCK, 4) k_search_bits(const JobDesc *jobs, SearchCtl C, int kmax) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    BitsWarp<KM> W;
    W.base = smem + wib * BitsLayout<KM>::BYTES;
    W.slab = C.slab + ((size_t)blockIdx.x * WARPS_PER_BLOCK + wib) * ((size_t)KM * NWL * 32);
    W.lcr = 0;
    int *M = W.M();
    uint64_t used[NWL];   // this lane's words of the used-vertex bitset (word lane + 32 w)

    const unsigned long long deadline = C.deadline_ns ? globaltimer() + C.deadline_ns : 0ull;
    Frame fr;
    unsigned iter = 0, last_don_iter = 0;
    unsigned long long last_check = 0, last_don_ns = 0, last_cancel = 0;
    int cur_job = -1;
    BitsJob B;
    WarpClock::begin(C);
    if (threadIdx.x == 0) atomicMax(C.span, ~globaltimer());
    while (acquire_frame(C, M, fr, deadline)) {
        WarpClock::frame_in(C);
        const JobDesc &J = jobs[fr.job];
        if (fr.job != cur_job) {
            // cache the job's pointers in registers and its position table in shared memory
            cur_job = fr.job;
            B.filt = J.filt; B.adj = J.t.adj; B.vld = J.t.vld; B.dw = J.t.dw; B.k = J.k;
            for (int t = lane; t < B.k; t += 32) {
                const PosInfo P = J.pos[t];
                PosB q;
                // back edges come in ascending position order, so one to position t - 1 is the last
                const bool prev_back = P.bcnt > 0 && J.back[P.bbeg + P.bcnt - 1].pos == t - 1;
                const bool prev_par = t > 0 && P.par == t - 1;
                q.pv = (int16_t)P.pv; q.par = (int16_t)P.par; q.bb = (int16_t)P.bbeg;
                q.bc = (int16_t)(P.bcnt - (prev_back ? 1 : 0));
                q.ucnt = (J.flags & JOB_RIDS) ? P.ucnt : J.t.n;   // RI: all of V_t
                q.abf = ((P.par >= 0 ? 2 : 1) + P.bcnt) * J.t.dw * 8 | (prev_back || prev_par ? PREV_ADJ : 0) |
                        (prev_par ? PREV_PAR : 0);
                W.tab()[t] = q;
            }
            __syncwarp();
            const int nb = J.pos[B.k - 1].bbeg + J.pos[B.k - 1].bcnt;
            for (int b = lane; b < nb; b += 32) W.tback()[b] = (uint8_t)J.back[b].pos;
            __syncwarp();
        }
        const int k = B.k, d0 = fr.depth;
        unsigned long long st = 0, nd = 0, mt = 0, hs = 0, ab = 0;   // the frame's totals
        unsigned st32 = 0, nd32 = 0, mt32 = 0, ab32 = 0;               // since the last fold
        {
#pragma unroll
            for (int w = 0; w < NWL; ++w) used[w] = 0ull;
            __syncwarp();
            for (int t = 0; t < d0; ++t) used_flip<NWL>(used, M[t]);
            if (lane == 0) M[d0] = -1;
            __syncwarp();
        }
        bool stopped = false;
        // a range frame covers candidates [beg, end) of its node: as the candidate
        // lists are ascending, that is the vertex-id interval [first, last]
        int vlo = 0, vhi = 0x7fffffff;
        bool counts = true;   // this part counts the node's states
        if (fr.beg >= 0) {
            const JobRef v{&J};
            const PosInfo *P = J.pos + d0;
            const PosV p = load_pos(P);
            // (a run's range as it stands; any other range counts in the plain list)
            const Cand S = fr.in_run ? pick_warp<false>(v, p, P, M) : plain_list<false>(v, p, P, M);
            int lo, hi, rb = 1, re = 1;
            counts = list_range<false>(v, p, S, M, fr.beg, fr.end, fr.in_run, lo, hi);
            if (lo < hi) row_range<false>(v, p, S, M, lo, hi, rb, re);
            if (lane == 0) { W.frange()[0] = rb; W.frange()[1] = re; }   // read back only by a checkpoint
            if (lo >= hi) { vlo = 1; vhi = 0; }
            else { vlo = cand_id(S, lo); vhi = cand_id(S, hi - 1); }
        } else if (lane == 0) {
            W.frange()[0] = W.frange()[1] = -1;
        }
        const bool count_len = counts && !fr.counted;
        const bool leaf0 = d0 == k - 1;
        int c0;
        {
            // the frame's first expansion: position d0 with M[0..d0-1] given and all in `used`
            const PosB p = W.tab()[d0];
            uint64_t s[NWL];
            int len;
            bits_rows<NWL, KM>(B, W, p, d0, true, used, s, len);
            if (count_len) st32 += (unsigned)len;
            ab32 += (unsigned)(p.abf & ABYTES_MASK);
            c0 = fr.beg >= 0 ? bits_finish<NWL, KM, true>(J, W, s, d0, p.pv, leaf0, hs, vlo, vhi)
                             : bits_finish<NWL, KM>(J, W, s, d0, p.pv, leaf0, hs);
        }
        if (!fr.counted) nd += c0;
        if (leaf0) {
            mt += c0;
        } else if (c0 > 0) {
            // Levels d0..lvl hold pending survivors; `used` holds M_0..M_{lvl-1} (not the
            // choice at lvl).  Pv is the part of position lvl + 1's candidate set that does
            // not depend on M[lvl] (see bits_rows), valid while `pok`: consecutive siblings
            // at one level share it, and a descent or ascent invalidates it.  An expansion
            // that finds no survivors does not descend, so a level's list is read only
            // after an expansion filled it.
            int lvl = d0;
            bool pok = false;
            uint64_t Pv[NWL];
            int plen = 0;
#pragma unroll
            for (int w = 0; w < NWL; ++w) Pv[w] = 0ull;
            for (;;) {
                if (((++iter) & 63) == 0) {
                  st += st32; nd += nd32; mt += mt32; ab += ab32;
                  st32 = nd32 = mt32 = ab32 = 0;
                  if (time_to_check(last_check)) {
                    if (C.budget > 0) {
                        if (lane == 0) atomicAdd(J.ctr + 1, st);
                        st = 0;
                    }
                    if (must_stop(C, J, st, deadline, last_check, last_cancel)) { stopped = true; break; }
                    if ((iter - last_don_iter >= (unsigned)C.donate_iters || last_check - last_don_ns >= C.donate_ns) &&
                        donation_claim(C)) {
                        // donate up to `gran` pending survivors of the shallowest level that has some
                        last_don_iter = iter;
                        last_don_ns = last_check;
                        const unsigned long long tdon = WarpClock::don_begin(C);
                        int given = 0;
                        for (int l = d0; l <= lvl && l + 1 + DONATE_MIN_LEVELS <= k; ++l) {
                            given = 0;
                            while (given < C.gran) {
                                const int v = bits_next<NWL, KM>(W, l);
                                if (v < 0) break;
                                if (!push_frame(C, fr.job, l + 1, -1, -1, M, l, v)) {
                                    bits_unnext<NWL, KM>(W, l, v);
                                    given = C.gran;
                                    break;
                                }
                                ++given;
                            }
                            if (given > 0) break;
                        }
                        WarpClock::don_end(C, tdon, given);
                        donation_done(C);
                    }
                  }
                }
                const int v = bits_next<NWL, KM>(W, lvl);
                if (v < 0) {
                    if (lvl == d0) break;
                    --lvl;
                    used_flip<NWL>(used, M[lvl]);   // the choice at the new current level leaves `used`
                    pok = false;
                    continue;
                }
                const int i = lvl + 1;
                const PosB p = W.tab()[i];
                if (!pok) {
                    bits_rows<NWL, KM>(B, W, p, i, false, used, Pv, plen);
                    pok = true;
                }
                uint64_t s[NWL];
#pragma unroll
                for (int w = 0; w < NWL; ++w) s[w] = Pv[w];
                int len = plen;
                if (p.abf & PREV_ADJ) {
                    and_row<NWL>(B.adj, B.dw, v, s);   // A[v] never holds v itself
                    if (p.abf & PREV_PAR) len = __ldg(B.vld + v).y;
                } else {
                    uint64_t nv[NWL];
#pragma unroll
                    for (int w = 0; w < NWL; ++w) nv[w] = ~0ull;
                    used_flip<NWL>(nv, v);
#pragma unroll
                    for (int w = 0; w < NWL; ++w) s[w] &= nv[w];
                }
                st32 += (unsigned)len;
                ab32 += (unsigned)(p.abf & ABYTES_MASK);
                const bool leaf = i == k - 1;
                if (leaf) {
                    // the match rows and the hash read M[0..i-1]: store the choice first when
                    // the set is not empty
                    int any = 0;
#pragma unroll
                    for (int w = 0; w < NWL; ++w) any |= s[w] != 0ull;
                    if (__any_sync(FULL, any)) {
                        if (lane == 0) M[lvl] = v;
                        __syncwarp();
                    }
                    const int c = bits_finish<NWL, KM>(J, W, s, i, p.pv, true, hs);
                    nd32 += c;
                    mt32 += c;
                } else {
                    const int c = bits_finish<NWL, KM>(J, W, s, i, p.pv, false, hs);
                    nd32 += c;
                    if (c > 0) {
                        if (lane == 0) M[lvl] = v;
                        __syncwarp();
                        used_flip<NWL>(used, v);
                        lvl = i;
                        pok = false;
                        continue;
                    }
                }
                // no descent: when that was the last survivor of its list, go up at once
                // (levels whose lists ran out) instead of finding out on the next iteration
                if (lvl > d0 && W.lc(lvl) == 0) {
                    do {
                        --lvl;
                        used_flip<NWL>(used, M[lvl]);
                    } while (lvl > d0 && W.lc(lvl) == 0);
                    pok = false;
                }
            }
            if (stopped && C.ckpt != nullptr) {
                // checkpoint: the pending survivors of each level as one counted range frame.
                // They are a contiguous run of the level's ascending survivors (a short list is
                // taken from its top, a spilled bitset from its lowest bit), so one index range
                // of the level's candidate list holds exactly them among the feasible candidates.
                for (int l = d0; l <= lvl; ++l) {
                    const PosB p = W.tab()[l];
                    const int32_t *lst = nullptr;
                    int len = J.t.n;
                    if (p.par >= 0) {
                        const int a = M[p.par];
                        const int b0 = __ldg(J.t.rowptr + a);
                        lst = J.t.col + b0;
                        len = __ldg(J.t.rowptr + a + 1) - b0;
                    } else if (J.flags & JOB_RIDS) {
                        lst = J.ulist + J.pos[l].uoff;
                        len = J.pos[l].ucnt;
                    }
                    int lo = 0, hi = len;   // the level's own range
                    if (l == d0 && W.frange()[0] >= 0) { lo = W.frange()[0]; hi = min(W.frange()[1], len); }
                    const int c = W.lc(l);
                    if (c == 0) continue;
                    if (c != LIST_SPILLED) {
                        const int vmax = W.lst()[l * W.LCAP + c - 1];
                        hi = lst ? lower_bound_warp(lst, len, vmax + 1) : vmax + 1;
                    } else {
                        const int vmin = bits_next<NWL, KM>(W, l);
                        if (vmin < 0) continue;
                        lo = lst ? lower_bound_warp(lst, len, vmin) : vmin;
                    }
                    if (lo < hi) ckpt_push(C, fr.job, l, true, lo, hi, M);
                }
            }
        }
        st += st32; nd += nd32; mt += mt32; ab += ab32;
        hs = warp_sum(hs);
        if (lane == 0) {
            atomicAdd(J.ctr + 0, mt);
            atomicAdd(J.ctr + 1, st);
            atomicAdd(J.ctr + 2, nd);
            atomicAdd(J.ctr + 3, hs);
            atomicAdd(J.abytes, ab);
            if (!stopped) atomicSub(C.outstanding, 1);
        }
        __syncwarp();
        WarpClock::frame_out(C, fr, st, nd);
        if (stopped) break;
    }
    WarpClock::finish(C);
    if ((threadIdx.x & 31) == 0) atomicMax(C.span + 1, globaltimer());
}

unsigned grid_for(long long warps) {
    long long blocks = (warps + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK;
    if (blocks < 1) blocks = 1;
    return (unsigned)blocks;
}

}  // namespace

// ================================================================ launchers

cudaError_t launch_domain_init_buckets(const JobDesc *jobs, const long long *vert_off, int njobs, long long nverts,
                                       cudaStream_t st) {
    if (nverts <= 0) return cudaSuccess;
    k_domain_init_buckets<<<dim3(grid_for(nverts), BUCKET_PARTS), BLOCK, 0, st>>>(jobs, vert_off, njobs, nverts);
    return cudaGetLastError();
}

cudaError_t launch_label_index(const JobDesc *jobs, int njobs, cudaStream_t st) {
    if (njobs <= 0) return cudaSuccess;
    k_label_index<<<njobs, KMAX, 0, st>>>(jobs);
    return cudaGetLastError();
}

cudaError_t launch_domain_init(const JobDesc *jobs, const long long *unit_off, int njobs, long long nunits,
                               cudaStream_t st) {
    if (nunits <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // words per warp: up to 32 (a warp steps along its words reading each job's and vertex's
    // fields once), fewer when that would leave the device short of warps (64 per SM)
    const long long want = nunits / ((long long)sms * 64);
    const int wpw = (int)std::max<long long>(1, std::min<long long>(INIT_WORDS_PER_WARP, want));
    k_domain_init<<<grid_for((nunits + wpw - 1) / wpw), BLOCK, 0, st>>>(jobs, unit_off, njobs, nunits, wpw);
    return cudaGetLastError();
}

cudaError_t launch_domain_ac(const JobDesc *jobs, const int4 *ent, const long long *eoff, int nent, long long nunits,
                             int *changed, unsigned char *vchanged, cudaStream_t st) {
    if (nunits <= 0) return cudaSuccess;
    k_domain_ac<<<grid_for(nunits), BLOCK, 0, st>>>(jobs, ent, eoff, nent, nunits, changed, vchanged);
    return cudaGetLastError();
}

cudaError_t launch_domain_ac_cand(const JobDesc *jobs, const int4 *ent, const long long *eoff, int nent,
                                  long long ncand, int32_t *cand, int *changed, unsigned char *vchanged,
                                  cudaStream_t st) {
    if (ncand <= 0) return cudaSuccess;
    const long long blocks = (ncand + BLOCK - 1) / BLOCK;
    k_domain_ac_cand<<<(unsigned)blocks, BLOCK, 0, st>>>(jobs, ent, eoff, nent, ncand, cand, changed, vchanged);
    return cudaGetLastError();
}

cudaError_t launch_domain_fc(const JobDesc *jobs, const long long *vert_off, const long long *sizes, int njobs,
                             int *changed, unsigned char *vchanged, cudaStream_t st) {
    if (njobs <= 0) return cudaSuccess;
    k_domain_fc<<<njobs, BLOCK, 0, st>>>(jobs, vert_off, sizes, changed, vchanged);
    return cudaGetLastError();
}

cudaError_t launch_domain_fixpoint(const JobDesc *jobs, int njobs, const long long *vert_off, const long long *cstart,
                                   const long long *csize, int32_t *cand, int *next_job, cudaStream_t st) {
    if (njobs <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // few pairs: one large block each, so that they still fill the device; many pairs:
    // blocks of four warps (eight pairs in flight per SM; 256 threads measured 3% slower and
    // 64 threads 15% slower on 196,000 molecule pairs), as many as are resident at once,
    // each taking pairs from the counter
    const int threads = njobs < sms * 4 ? FIXPOINT_BIG_BLOCK : FIXPOINT_SMALL_BLOCK;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_domain_fixpoint, threads, 0);
    if (e != cudaSuccess) return e;
    const long long wave = (long long)sms * std::max(occ, 1);
    const int grid = (int)std::min<long long>(njobs, wave);
    e = cudaMemsetAsync(next_job, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    k_domain_fixpoint<<<grid, threads, 0, st>>>(jobs, njobs, vert_off, cstart, csize, cand, next_job);
    return cudaGetLastError();
}

cudaError_t launch_domain_fixpoint_warp(const JobDesc *jobs, int njobs, const WarpFixpoint &W, cudaStream_t st) {
    if (njobs <= 0) return cudaSuccess;
    if (W.nmax > WARP_FP_N || W.classes > WARP_FP_CLASSES || (W.nmax & 31)) return cudaErrorInvalidValue;
    const int smem = WARPS_PER_BLOCK * warp_fixpoint_smem(W.nmax, W.classes);
    int dev = 0, sms = 0, occ = 0;
    // (the attribute is the function's, for every thread of the process: always the largest launch's)
    cudaError_t e = cudaFuncSetAttribute(k_domain_fixpoint_warp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         WARPS_PER_BLOCK * warp_fixpoint_smem(WARP_FP_N, WARP_FP_CLASSES));
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_domain_fixpoint_warp, BLOCK, smem);
    if (e == cudaSuccess) e = cudaMemsetAsync(W.next, 0, 16, st);
    if (e != cudaSuccess) return e;
    const int grid = std::min((njobs + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK, sms * std::max(occ, 1));
    k_domain_fixpoint_warp<<<grid, BLOCK, smem, st>>>(jobs, njobs, W);
    return cudaGetLastError();
}
bool domain_fixpoint_warp_fits(int k, int n, int classes) {
    return k <= WARP_FP_K && n <= WARP_FP_N && classes <= WARP_FP_CLASSES;
}

size_t domain_coop_bytes(long long nverts, long long nedges) {
    return 128 + (size_t)nverts * (sizeof(CoopVert) + 4 + 3 + 1) + (size_t)nedges * sizeof(CoopEdge) + 64;
}

cudaError_t launch_domain_coop(const JobDesc *jobs, const long long *vert_off, const int *edge_off, int njobs,
                               long long nverts, long long nedges, int any_fc, int longest_list, void *scratch,
                               int *slots, long long cap, int blocks_per_sm, cudaStream_t st) {
    if (nverts <= 0) return cudaSuccess;
    if (nverts > DOMAIN_COOP_VERTS) return cudaErrorInvalidValue;
    DomainCoop D;
    D.jobs = jobs; D.vert_off = vert_off; D.edge_off = edge_off; D.njobs = njobs; D.nverts = (int)nverts;
    D.any_fc = any_fc;
    D.any_long = longest_list > AC_WARP_LIST;
    char *b = static_cast<char *>(scratch);
    D.status = reinterpret_cast<int *>(b);
    D.bar = reinterpret_cast<unsigned *>(b) + 1;
    D.any = reinterpret_cast<int *>(b) + 4;
    D.nheavy = reinterpret_cast<int *>(b) + 8;
    b += 128;
    D.size = reinterpret_cast<int *>(b); b += 4 * nverts;
    D.chg = reinterpret_cast<unsigned char *>(b); b += 3 * nverts;
    D.done = reinterpret_cast<unsigned char *>(b); b += nverts;
    const size_t zeroed = (size_t)(b - static_cast<char *>(scratch));
    b = static_cast<char *>(scratch) + ((zeroed + 15) & ~(size_t)15);
    D.vert = reinterpret_cast<CoopVert *>(b); b += nverts * sizeof(CoopVert);
    D.edge = reinterpret_cast<CoopEdge *>(b);
    D.slot = reinterpret_cast<int2 *>(slots);
    D.heavy = slots + 2 * cap;
    D.cap = cap;
    cudaError_t e = cudaMemsetAsync(scratch, 0, zeroed, st);
    if (e != cudaSuccess) return e;
    const size_t smem = ((size_t)nverts + 1) * sizeof(int);
    int dev = 0, sms = 0, occ = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_domain_coop, BLOCK, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    void *args[] = {(void *)&D};
    const int per_sm = std::min(occ, blocks_per_sm > 0 ? blocks_per_sm : DOMAIN_COOP_BLOCKS);
    return cudaLaunchCooperativeKernel((void *)k_domain_coop, dim3(sms * per_sm), dim3(BLOCK), args, smem, st);
}

cudaError_t launch_domain_sizes(const JobDesc *jobs, const long long *vert_off, int njobs, long long nverts,
                                long long *sizes, cudaStream_t st) {
    if (nverts <= 0) return cudaSuccess;
    k_domain_sizes<<<grid_for(nverts), BLOCK, 0, st>>>(jobs, vert_off, njobs, nverts, sizes);
    return cudaGetLastError();
}

cudaError_t launch_domain_lists(const JobDesc *jobs, const int *task_job, const int *task_vert, const int *task_out,
                                int ntasks, int32_t *lists, cudaStream_t st) {
    if (ntasks <= 0) return cudaSuccess;
    k_domain_lists<<<ntasks, BLOCK, 0, st>>>(jobs, task_job, task_vert, task_out, lists);
    return cudaGetLastError();
}

cudaError_t launch_split(const JobDesc *jobs, const int32_t *fin, long long nf, int depth, int32_t *counts,
                         const long long *offs, int32_t *fout, int pass, int count_ctr, int directed,
                         cudaStream_t st) {
    if (nf <= 0) return cudaSuccess;
    long long warps = nf;
    if (warps > 152LL * 64) warps = 152LL * 64;
    if (directed)
        k_split<true><<<grid_for(warps), BLOCK, 0, st>>>(jobs, fin, nf, depth, counts, offs, fout, pass, count_ctr);
    else
        k_split<false><<<grid_for(warps), BLOCK, 0, st>>>(jobs, fin, nf, depth, counts, offs, fout, pass, count_ctr);
    return cudaGetLastError();
}

cudaError_t launch_split_coop(const JobDesc *jobs, long long f0, int32_t *buf0, int32_t *buf1, long long cap_ints,
                              long long target, int max_levels, long long *wtot, long long wtot_cap,
                              unsigned *bar, long long *result, int *status, int count_ctr, int directed,
                              int blocks_per_sm, uint32_t *masks, long long mask_total, int ordered,
                              const SplitAsync &async, long long *trace, cudaStream_t st) {
    SplitCtl S;
    S.narrow = ordered ? 0 : async.narrow;
    unsigned long long *aw = static_cast<unsigned long long *>(async.ctl);   // one line each, zeroed
    S.qhead = aw; S.qtail = aw + 16; S.pend = reinterpret_cast<long long *>(aw + 32); S.top = aw + 48;
    S.nleft = aw + 64; S.stop = reinterpret_cast<int *>(aw + 80);
    S.qentry = async.entries; S.qcap = async.qcap; S.epoch = async.epoch;
    S.left = async.left;
    S.trace = ordered ? nullptr : trace;
    S.buf0 = buf0; S.buf1 = buf1; S.cap_ints = cap_ints; S.target = target; S.max_levels = max_levels;
    S.wtot = wtot; S.bar = bar; S.result = result; S.status = status; S.count_ctr = count_ctr;
    S.masks = masks; S.mask_total = masks ? mask_total : 0;
    int dev = 0, sms = 0, occ = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    void *fn = ordered ? (directed ? (void *)k_split_coop<true> : (void *)k_split_coop<false>)
                       : (directed ? (void *)k_split_once<true> : (void *)k_split_once<false>);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, BLOCK, 0);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    if (blocks_per_sm > 0 && blocks_per_sm < occ) occ = blocks_per_sm;
    if ((long long)sms * occ * WARPS_PER_BLOCK > wtot_cap) occ = (int)(wtot_cap / ((long long)sms * WARPS_PER_BLOCK));
    if (occ < 1) return cudaErrorInvalidConfiguration;
    // all blocks must be co-resident for the grid barrier: a cooperative launch guarantees it
    dim3 grid(sms * occ), block(BLOCK);
    void *args[] = {(void *)&jobs, (void *)&f0, (void *)&S};
    return cudaLaunchCooperativeKernel(fn, grid, block, args, 0, st);
}

size_t scan_tmp_bytes(long long n) {
    const long long tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    return (size_t)(tiles + 1) * sizeof(long long);
}

cudaError_t launch_scan(const int32_t *in, long long *out, long long n, long long *total, void *tmp, size_t tmp_bytes,
                        cudaStream_t st) {
    const long long tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    if ((size_t)(tiles + 1) * sizeof(long long) > tmp_bytes) return cudaErrorInvalidValue;
    long long *tile_sum = static_cast<long long *>(tmp);
    if (n <= 0) {
        return cudaMemsetAsync(total, 0, sizeof(long long), st);
    }
    k_scan_tiles<<<(unsigned)tiles, BLOCK, 0, st>>>(in, out, n, tile_sum);
    k_scan_sums<<<1, BLOCK, 0, st>>>(tile_sum, tiles, total);
    k_scan_add<<<(unsigned)tiles, BLOCK, 0, st>>>(out, n, tile_sum);
    return cudaGetLastError();
}

int search_warps_per_block() { return WARPS_PER_BLOCK; }

namespace {
// One block per hub: set the bit of every neighbour in the hub's row.
__global__ void k_build_hubs(const int32_t *rowptr, const int32_t *col, const int32_t *hubs, int dw, uint64_t *bits) {
    const int x = hubs[blockIdx.x];
    uint64_t *row = bits + (size_t)blockIdx.x * dw;
    for (int e = rowptr[x] + threadIdx.x; e < rowptr[x + 1]; e += blockDim.x) {
        const int y = col[e];
        atomicOr((unsigned long long *)(row + (y >> 6)), 1ull << (y & 63));
    }
}
}  // namespace

cudaError_t launch_frames_to_rows(const JobDesc *jobs, int32_t *frames, long long n, long long pitch,
                                  const unsigned long long *seq, int directed, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (directed) k_frames_to_rows<true><<<grid_for(n), BLOCK, 0, st>>>(jobs, frames, n, pitch, seq);
    else k_frames_to_rows<false><<<grid_for(n), BLOCK, 0, st>>>(jobs, frames, n, pitch, seq);
    return cudaGetLastError();
}

cudaError_t launch_build_hubs(const int32_t *rowptr, const int32_t *col, const int32_t *hubs, int h, int dw,
                              uint64_t *bits, cudaStream_t st) {
    if (h <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(bits, 0, (size_t)h * dw * sizeof(uint64_t), st);
    if (e != cudaSuccess) return e;
    k_build_hubs<<<h, BLOCK, 0, st>>>(rowptr, col, hubs, dw, bits);
    return cudaGetLastError();
}

namespace {
__global__ void k_pool_init(unsigned long long *seq, int cap) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < cap; i += gridDim.x * blockDim.x)
        seq[i] = (unsigned long long)i;
}
}  // namespace

cudaError_t launch_pool_init(unsigned long long *seq, int cap, cudaStream_t st) {
    k_pool_init<<<(cap + BLOCK - 1) / BLOCK, BLOCK, 0, st>>>(seq, cap);
    return cudaGetLastError();
}

// ------------------------------------------------------- records of a huge batch
//
// A plain RI batch of many pairs repeats few targets and patterns, so its job records (368 bytes
// each) and root frames are put together here from per-graph tables and 12 bytes per pair: one warp
// writes one record, its words spread over the lanes.  Bound by the record writes (200,000
// pairs: 74 MB; written by 16 host threads, uploaded, and given their roots by one, they took
// 4.5 ms of a 9.7 ms call, now 5.3 ms).
namespace {
__global__ void __launch_bounds__(BLOCK) k_build_jobs(JobTables T) {
    __shared__ JobDesc rec[WARPS_PER_BLOCK];
    const int lane = threadIdx.x & 31;
    JobDesc &D = rec[threadIdx.x >> 5];
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long q = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < T.nj; q += nw) {
        const int2 pair = T.pair[q];
        const TargetView *t = T.target + pair.x;
        const PatternRow *p = T.pattern + pair.y;
        static_assert(sizeof(TargetView) % 4 == 0 && sizeof(PatternView) % 4 == 0 && sizeof(JobDesc) % 4 == 0, "copied as words");
        for (int i = lane; i < (int)(sizeof(TargetView) / 4); i += 32)
            reinterpret_cast<int *>(&D.t)[i] = reinterpret_cast<const int *>(t)[i];
        for (int i = lane; i < (int)(sizeof(PatternView) / 4); i += 32)
            reinterpret_cast<int *>(&D.p)[i] = reinterpret_cast<const int *>(&p->view)[i];
        __syncwarp();
        const int n = D.t.n, k = D.p.k;
        if (lane == 0) {
            const bool longl = D.t.maxdeg == 0 || D.t.maxdeg > SPLIT_RANGE || (p->unparented && n > SPLIT_RANGE);
            D.pos = p->pos;
            D.back = p->back;
            D.filt = nullptr;
            D.ulist = nullptr;
            D.plidx = nullptr;
            D.k = k;
            D.flags = T.flags | (longl ? JOB_LONG_LISTS : 0);
            D.ctr = T.ctr + 4 * q;
            D.mbuf = nullptr;
            D.mcap = 0;
            D.mlen = T.ctr + 4 * T.nj + q;
            D.abytes = T.ctr + 5 * T.nj + q;
        }
        __syncwarp();
        for (int i = lane; i < (int)(sizeof(JobDesc) / 4); i += 32)
            reinterpret_cast<int *>(T.out + q)[i] = reinterpret_cast<const int *>(&D)[i];
        // its root frames: the whole list, or ranges of `chunk` candidates
        const int r0 = T.root_off[q], r1 = T.root_off[q + 1];
        for (int r = r0 + lane; r < r1; r += 32) {
            const int b = r1 - r0 == 1 ? -1 : (r - r0) * T.chunk;
            reinterpret_cast<int4 *>(T.roots)[r] = make_int4((int)q, 0, b, b < 0 ? -1 : min(b + T.chunk, n));
        }
        __syncwarp();
    }
}
}  // namespace

cudaError_t launch_build_jobs(const JobTables &T, cudaStream_t st) {
    if (T.nj <= 0) return cudaSuccess;
    k_build_jobs<<<(unsigned)std::min<long long>((T.nj + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK, 1 << 16), BLOCK, 0, st>>>(T);
    return cudaGetLastError();
}

// ------------------------------------------------------- listed matches
//
// Listed matches come out in the order their warps found them; the caller gets them sorted by the
// images of pattern vertices 0, 1, ...  A merge sort of row numbers under their first two images
// (one 64-bit key, beside the number; the row itself is read only where keys tie): tiles of
// MATCH_TILE by a bitonic network in shared memory, then passes that merge runs pairwise, each element
// finding its place by a binary search of the other run (rows are distinct, so no two meet).
// Bound by the searches' dependent loads and the launches: listing some 15,000 matches of 6
// vertices takes 0.48 ms a call, 0.26 of it the search, where numpy's lexsort of the columns on the
// host and a count to size the buffer made it 2.8 ms.
namespace {

constexpr int MATCH_TILE = 1024;

// Row a before row b?
__device__ __forceinline__ bool match_before(uint64_t ka, uint32_t a, uint64_t kb, uint32_t b, const int32_t *rows, int k) {
    if (ka != kb) return ka < kb;
    const int32_t *ra = rows + (size_t)a * k, *rb = rows + (size_t)b * k;
    for (int i = 2; i < k; ++i) {
        const int x = __ldg(ra + i), y = __ldg(rb + i);
        if (x != y) return x < y;
    }
    return a < b;   // (the padding of a tile)
}

__global__ void __launch_bounds__(MATCH_TILE / 2) k_match_tiles(const int32_t *rows, long long n, int k, uint64_t *key,
                                                                uint32_t *row) {
    __shared__ uint64_t sk[MATCH_TILE];
    __shared__ uint32_t sr[MATCH_TILE];
    const long long base = (long long)blockIdx.x * MATCH_TILE;
    const int m = (int)min((long long)MATCH_TILE, n - base);
    for (int i = threadIdx.x; i < MATCH_TILE; i += MATCH_TILE / 2) {
        sk[i] = ~0ull;   // (padding sorts last: images are not negative)
        sr[i] = (uint32_t)(base + i);
        if (i < m) {
            const int32_t *r = rows + (size_t)(base + i) * k;
            sk[i] = (uint64_t)(uint32_t)r[0] << 32 | (k > 1 ? (uint32_t)r[1] : 0u);
        }
    }
    for (int size = 2; size <= MATCH_TILE; size <<= 1)
        for (int step = size >> 1; step >= 1; step >>= 1) {
            __syncthreads();
            const int a = 2 * step * (threadIdx.x / step) + threadIdx.x % step, b = a + step;
            const bool up = (a & size) == 0;
            const uint64_t ka = sk[a], kb = sk[b];
            const uint32_t ra = sr[a], rb = sr[b];
            // (rows beyond the list never tie with one of it, and among themselves order does not matter)
            const bool swap = ka == kb && ka == ~0ull ? (rb < ra) == up : match_before(kb, rb, ka, ra, rows, k) == up;
            if (swap) {
                sk[a] = kb; sk[b] = ka;
                sr[a] = rb; sr[b] = ra;
            }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += MATCH_TILE / 2) {
        key[base + i] = sk[i];
        row[base + i] = sr[i];
    }
}

// Runs of `width` merged pairwise.
__global__ void __launch_bounds__(BLOCK) k_match_merge(const int32_t *rows, long long n, int k, long long width,
                                                       const uint64_t *key, const uint32_t *row, uint64_t *okey,
                                                       uint32_t *orow) {
    for (long long i = blockIdx.x * (long long)BLOCK + threadIdx.x; i < n; i += (long long)gridDim.x * BLOCK) {
        const long long pair = i / (2 * width) * (2 * width), mid = min(pair + width, n), end = min(pair + 2 * width, n);
        const uint64_t ki = key[i];
        const uint32_t ri = row[i];
        const bool first = i < mid;
        long long lo = first ? mid : pair, hi = first ? end : mid;
        const long long from = lo;
        while (lo < hi) {   // elements of the other run before this one
            const long long m = (lo + hi) >> 1;
            if (match_before(key[m], row[m], ki, ri, rows, k)) lo = m + 1; else hi = m;
        }
        const long long at = pair + (i - (first ? pair : mid)) + (lo - from);
        okey[at] = ki;
        orow[at] = ri;
    }
}

__global__ void __launch_bounds__(BLOCK) k_match_gather(const int32_t *rows, long long n, int k, const uint32_t *row,
                                                        int32_t *out) {
    for (long long i = blockIdx.x * (long long)BLOCK + threadIdx.x; i < n * k; i += (long long)gridDim.x * BLOCK) {
        const long long r = i / k;
        out[i] = rows[(size_t)row[r] * k + (i - r * k)];
    }
}

}  // namespace

size_t match_sort_bytes(long long n) { return (size_t)n * 2 * (sizeof(uint64_t) + sizeof(uint32_t)); }

cudaError_t launch_match_sort(const int32_t *rows, long long n, int k, void *scratch, int32_t *out, int *launches,
                              cudaStream_t st) {
    if (n <= 0 || k <= 0) return cudaSuccess;
    if (n > UINT32_MAX) return cudaErrorInvalidValue;
    uint64_t *key[2] = {static_cast<uint64_t *>(scratch), static_cast<uint64_t *>(scratch) + n};
    uint32_t *row[2] = {reinterpret_cast<uint32_t *>(key[1] + n), reinterpret_cast<uint32_t *>(key[1] + n) + n};
    auto blocks = [](long long items) { return (unsigned)std::min<long long>((items + BLOCK - 1) / BLOCK, 1 << 20); };
    k_match_tiles<<<(unsigned)((n + MATCH_TILE - 1) / MATCH_TILE), MATCH_TILE / 2, 0, st>>>(rows, n, k, key[0], row[0]);
    ++*launches;
    int cur = 0;
    for (long long w = MATCH_TILE; w < n; w *= 2, cur ^= 1, ++*launches)
        k_match_merge<<<blocks(n), BLOCK, 0, st>>>(rows, n, k, w, key[cur], row[cur], key[cur ^ 1], row[cur ^ 1]);
    k_match_gather<<<blocks(n * k), BLOCK, 0, st>>>(rows, n, k, row[cur], out);
    ++*launches;
    return cudaGetLastError();
}

size_t search_smem_bytes(int kernel, int kmax, int nwl) {
    return WARPS_PER_BLOCK * (kernel == 2 ? bits_smem_per_warp(kmax, nwl) : csr_smem_per_warp(kmax));
}

size_t search_slab_bytes(int kernel, int kmax, int nwl, long long grid) {
    if (kernel != 2) return 0;
    return (size_t)grid * WARPS_PER_BLOCK * bits_slab_words_per_warp(kmax, nwl) * sizeof(uint64_t);
}

// Let kernel `kern` take `smem` bytes of dynamic shared memory.  The limit is
// a property of the kernel shared by every host thread that launches it, so
// it is always raised to the device maximum, never set to one launch's need:
// concurrent launches of different sizes (serving groups) cannot lower it
// under one another.
template <typename K>
static cudaError_t allow_dynamic_smem(K kern, size_t smem) {
    if (smem <= 48 * 1024) return cudaSuccess;
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if ((long long)smem > optin) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
}

template <typename K>
static cudaError_t occupancy_of(K kern, size_t smem, int *occ) {
    cudaError_t e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kern, BLOCK, smem);
}

// f(kernel) of the bitset search for this pattern size and words per lane.
template <typename F>
static cudaError_t with_bits_kernel(int kmax, int nwl, F f) {
    switch (nwl * 1000 + bits_km(kmax)) {
        case 1024: return f(k_search_bits<1, 24>);
        case 1032: return f(k_search_bits<1, 32>);
        case 1064: return f(k_search_bits<1, 64>);
        case 1000 + KMAX: return f(k_search_bits<1, KMAX>);
        case 2024: return f(k_search_bits<2, 24>);
        case 2032: return f(k_search_bits<2, 32>);
        case 2064: return f(k_search_bits<2, 64>);
        case 2000 + KMAX: return f(k_search_bits<2, KMAX>);
        case 3024: return f(k_search_bits<3, 24>);
        case 3032: return f(k_search_bits<3, 32>);
        case 3064: return f(k_search_bits<3, 64>);
        case 3000 + KMAX: return f(k_search_bits<3, KMAX>);
        case 4024: return f(k_search_bits<4, 24>);
        case 4032: return f(k_search_bits<4, 32>);
        case 4064: return f(k_search_bits<4, 64>);
        case 4000 + KMAX: return f(k_search_bits<4, KMAX>);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t search_blocks_per_sm(int kernel, int kmax, int nwl, int directed, int *occ) {
    const size_t smem = search_smem_bytes(kernel, kmax, nwl);
    if (kernel == 2) return with_bits_kernel(kmax, nwl, [&](auto kern) { return occupancy_of(kern, smem, occ); });
    if (directed) return occupancy_of(k_search_csr<true>, smem, occ);
    return occupancy_of(k_search_csr<false>, smem, occ);
}

template <typename K>
static cudaError_t launch_persistent(K kern, const JobDesc *jobs, const SearchCtl &ctl, int kmax, size_t smem,
                                     int blocks_per_sm, long long max_grid, int *grid_out, cudaStream_t st) {
    int dev = 0, sms = 0, occ = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, BLOCK, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    int per_sm = (blocks_per_sm > 0 && blocks_per_sm < occ) ? blocks_per_sm : occ;
    long long g = (long long)sms * per_sm;
    if (max_grid > 0 && g > max_grid) g = max_grid;   // never more blocks than the scratch slab covers
    const int grid = (int)g;
    if (grid_out) *grid_out = grid;
    kern<<<grid, BLOCK, smem, st>>>(jobs, ctl, kmax);
    return cudaGetLastError();
}

cudaError_t launch_search(int kernel, const JobDesc *jobs, const SearchCtl &ctl, int kmax, int nwl, int directed,
                          int blocks_per_sm, long long max_grid, int *grid_out, cudaStream_t st) {
    const size_t smem = search_smem_bytes(kernel, kmax, nwl);
    if (kernel == 2)
        return with_bits_kernel(kmax, nwl, [&](auto kern) {
            return launch_persistent(kern, jobs, ctl, kmax, smem, blocks_per_sm, max_grid, grid_out, st);
        });
    if (directed) return launch_persistent(k_search_csr<true>, jobs, ctl, kmax, smem, blocks_per_sm, max_grid, grid_out, st);
    return launch_persistent(k_search_csr<false>, jobs, ctl, kmax, smem, blocks_per_sm, max_grid, grid_out, st);
}

}  // namespace sge
