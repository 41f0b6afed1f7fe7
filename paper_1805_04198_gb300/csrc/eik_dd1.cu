// eik_dd1.cu -- the one-dimensional two-scale iteration of Sec. 3.1 (Steps
// 1-4): eq. 1d on [0, 1] with the coarse grid X_i = i H (i = 0..N) and the
// subintervals [iH, (i+1)H] of M fine cells each (h = H / M).  eik_dd_solve
// runs it when grid->ndim == 1.
//
// One cooperative launch runs the whole iteration.  The subintervals are
// spread over one CTA per SM (a few consecutive subintervals per CTA, eight
// lanes each): the 1-D FSM of Sec. 1.1 (Steps 2-3) is a chain of dependent
// updates, bound by the latency of one FP64 addition and comparison per node
// where the wave passes; what it does not change is checked by all eight lanes
// at once (1024 subintervals of 1001 FP64 nodes, two iterations: 1.17 ms; one
// thread per subinterval, comparisons on the FP64 pipe: 6.5 ms).  CTA 0 holds the
// coarse state (U, the new U, u^k, C_H(U^k), the winds W^k and w^k, the fixed-node
// mask) in shared memory and runs the coarse work between two grid barriers: the
// Step 3 choice at the coarse nodes (its threads), then one warp for the serial
// part (Step 1's coarse FSM, Step 4's weighted Gauss-Seidel sweeps, the causal
// sweep, the update size), in the same form.  U and W are published to global
// memory for the next fine phase; the subintervals' end copies come back through
// global memory.
// Every grid barrier is a bounded wait: on expiry the kernel records
// EIK_EDEVICE_TIMEOUT in the statistics and returns.
//
// Readings, the same as for the 2-D method: a wind is the direction of travel
// (+1 when the left neighbour gives the minimum, so the W~ of Step 4 is read
// with the opposite sign to the printed one); a tie goes to the right
// neighbour; an inflow end of a subinterval starts at U and is swept like any
// node, and an end that keeps that starting value echoes the coarse wind and
// is no candidate of the minimum unless both copies are echoes; the weighted
// update is u^k + theta (U~ - C_H(U^k)), and u^k where U~ or C_H(U^k) is
// +inf; the causal sweep repeats both directions until nothing changes.
// Step 1 has no causal sweep (the 1-D text gives none), the Step 3 choice
// compares the two fine winds only, and Step 4 tests W^k = w^k = W~.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "engine.cuh"  // MAX_SWEEPS, the sweep cap of every DD solve
#include "host_util.h"
#include "prof.h"

namespace eik {

EIK_SPIN_LIMIT_SETTER(set_spin_limit_dd1)

constexpr int DD1_MAX_SUB = 2048;  // subintervals: the coarse state must fit in shared memory
constexpr int DD1_G = 8;           // lanes per subinterval
constexpr int DD1_THREADS = 512;   // at most: 64 subintervals on a CTA (a device of 32 SMs)

// Control words at the start of the workspace (cleared before every launch).
struct DD1Ctl {
    unsigned bar[2];  // grid barrier: arrivals, generation
    int err;          // EIK_OK or DEV_TIMEOUT
    int stop;         // set by CTA 0: 1 = the iteration ends after this fine phase
    unsigned long long fsm_max, fsm_caps, fine_upd;
};

template <class T>
struct DD1Args {
    const T *r;
    const uint8_t *gamma;
    const T *g;
    T *u;
    eik_dd_stats *stats;
    DD1Ctl *ctl;
    T *gU;            // U^k published for the fine phase (N + 1)
    int8_t *gW;       // W^k (N + 1)
    T *geu;           // end copies of the subintervals: 2 sub (left), 2 sub + 1 (right)
    int8_t *gew;      // their winds
    uint8_t *gee;     // their echo flags
    int N;            // subintervals
    int per;          // subintervals per CTA
    long long M;      // fine cells per subinterval
    T h, H, theta, tol;
    int max_iter;
    long long max_fsm, max_coarse;
};

// Shared memory of CTA 0: U, the new U, u^k, C_H(U^k), r(X_i) H (N + 1
// each), W^k, w^k and the fixed-node mask (N + 1 bytes each).
template <class T>
__host__ __device__ inline size_t dd1_coarse_bytes(int N) {
    return ((size_t)5 * (N + 1) * sizeof(T) + (size_t)3 * (N + 1) + 15) & ~(size_t)15;
}
// Nodes from one subinterval's values (or r h) in shared memory to the next: 8
// more than a multiple of 16, so that neighbouring groups use other banks.
__host__ __device__ inline long long dd1_pitch(long long M) { return (M + 16) / 16 * 16 + 8; }

static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

template <class T>
static size_t dd1_ws_bytes(int N) {
    return al256(sizeof(DD1Ctl)) + al256((size_t)(N + 1) * sizeof(T)) + al256((size_t)(N + 1)) +
           al256((size_t)2 * N * sizeof(T)) + al256((size_t)2 * N) + al256((size_t)2 * N);
}

// C_H of eq. 1dgod from the two neighbour values, with the wind of the one
// used (+1 left, -1 right, 0 when the value is +inf).  The 1-D Godunov update
// of a fine node is the same expression with spacing h.
template <class T>
__device__ __forceinline__ T ch1(T a, T b, T rh, int &w) {
    T v;
    if (a < b) {
        v = Num<T>::add(a, rh);
        w = 1;
    } else {
        v = Num<T>::add(b, rh);
        w = -1;
    }
    if (!(v < Num<T>::inf())) w = 0;
    return v;
}

template <class T>
__device__ __forceinline__ T ch1_at(const T *U, int i, int N, T rH, int &w) {
    const T inf = Num<T>::inf();
    return ch1(i > 0 ? U[i - 1] : inf, i < N ? U[i + 1] : inf, rH, w);
}

template <class T>
__device__ __forceinline__ T abs_(T x) {
    return x < T(0) ? -x : x;
}
__device__ __forceinline__ bool same_bits(float a, float b) { return __float_as_int(a) == __float_as_int(b); }
__device__ __forceinline__ bool same_bits(double a, double b) { return bits64(a) == bits64(b); }
__device__ __forceinline__ bool finite_(float a) { return (__float_as_int(a) & 0x7f800000) != 0x7f800000; }
__device__ __forceinline__ bool finite_(double a) { return (__double2hiint(a) & 0x7ff00000) != 0x7ff00000; }

// The Gauss-Seidel sweeps of this file.  A serial sweep sets v(p) = f(p, v(p - 1),
// old(p + 1)) at position p, one chain of dependent updates.  Most positions of
// most sweeps (those that the wave has passed or not reached, all of the last
// sweep) keep their values, and that can be seen for many of them at once: if
// f(p, old(p - 1), old(p + 1)) = old(p) at every position of a block whose
// predecessor kept its value, the serial sweep changes nothing there.  A block
// where that fails is walked node by node, with everything that does not depend
// on the node behind taken out of the chain.

// Whether a lane of this lane's group of DD1_G has p set.
__device__ __forceinline__ bool group_any(bool p) {
    return ((__ballot_sync(FULL, p) >> (threadIdx.x & 31 & ~(DD1_G - 1))) & ((1u << DD1_G) - 1)) != 0;
}

// Node of a plain sweep: v = min(old, min(neighbours) + r h); r h is NaN at Gamma
// (and where it is no finite number), which changes nothing.  Rounding is
// monotone, so min(behind, ahead) + r h is the smaller of the two sums, and only
// one of them is in the chain.
template <class T>
__device__ __forceinline__ T fsm_rest(T old, T rh, T ahead) {
    return Num<T>::mn(Num<T>::add(ahead, rh), old);
}
template <class T>
__device__ __forceinline__ T fsm_chain(T rest, T rh, T behind) {
    return Num<T>::mn(Num<T>::add(behind, rh), rest);
}

// One sweep over the N + 1 coarse nodes in direction DIR by one warp; returns
// whether a value changed.  load(j, x) gives node j (x.old its value), f(x,
// behind, ahead) its update, link(x, behind) the update of a node that follows
// the one behind it.  A lane has one of 32 nodes.  First every node takes its
// predecessor as it was, then as the first pass left it; if the two agree, they
// are the serial sweep's values.  Else the chain is added up on all lanes alike
// as if every node but the first followed its predecessor, the operands loaded
// ahead of it, and each lane checks its own node against the value behind it.
// Only if one did not follow are the nodes walked with f in the chain.
template <int DIR, class T, class Node, class Load, class Link, class F>
__device__ bool coarse_sweep(int n, T *v, Load load, Link link, F f) {
    constexpr int RUN = 8;
    const int lane = threadIdx.x & 31;
    const T inf = Num<T>::inf();
    auto at = [&](int p) { return DIR > 0 ? p : n - 1 - p; };
    auto value = [&](int p) { return p >= 0 && p < n ? v[at(p)] : inf; };
    bool ch = false;
#pragma unroll 1
    for (int p0 = 0; p0 < n; p0 += 32) {
        // (lanes past the end repeat the last node and count for nothing)
        const int p = min(p0 + lane, n - 1);
        const bool mine = p0 + lane < n;
        Node x;
        load(at(p), x);
        const T carry = value(p0 - 1), ahead = value(p + 1);
        auto update = [&](T of) {  // this lane's node after the values `of` of the lanes
            T behind = __shfl_up_sync(FULL, of, 1);
            if (lane == 0) behind = carry;
            return f(x, behind, ahead);
        };
        T nv = update(x.old);
        if (!__any_sync(FULL, mine && !same_bits(nv, x.old))) continue;
        T check = update(nv);
        if (__any_sync(FULL, mine && !same_bits(check, nv))) {
            const int count = min(32, n - p0);
            T t = __shfl_sync(FULL, nv, 0);  // (right already)
#pragma unroll 1
            for (int q = 1; q < count; q += RUN) {
                Node y[RUN];
#pragma unroll
                for (int i = 0; i < RUN; ++i) load(at(min(p0 + q + i, n - 1)), y[i]);
#pragma unroll
                for (int i = 0; i < RUN; ++i) {
                    t = link(y[i], t);
                    if (lane == q + i) nv = t;
                }
            }
            check = update(nv);
            if (__any_sync(FULL, mine && !same_bits(check, nv))) {
                t = carry;
#pragma unroll 1
                for (int q = 0; q < count; ++q) {
                    Node y;
                    load(at(min(p0 + q, n - 1)), y);
                    t = f(y, t, value(p0 + q + 1));
                    if (lane == q) nv = t;
                }
            }
        }
        __syncwarp();  // every lane has read what is overwritten now
        if (mine) {
            ch = ch || !(nv == x.old);
            v[at(p)] = nv;
        }
        __syncwarp();
    }
    return __any_sync(FULL, ch);
}

// Sweeps alternate right-to-left, left-to-right until one changes nothing or the
// cap is reached; the sweeps run.
template <class T, class Node, class Load, class Link, class Down, class Up>
__device__ long long coarse_sweeps(const DD1Args<T> &A, T *v, Load load, Link link, Down down, Up up, bool &conv) {
    long long s = 0;
    conv = false;
    while (s < A.max_coarse) {
        const bool ch = (s % 2 == 0) ? coarse_sweep<-1, T, Node>(A.N + 1, v, load, link, down)
                                     : coarse_sweep<1, T, Node>(A.N + 1, v, load, link, up);
        ++s;
        if (!ch) {
            conv = true;
            break;
        }
    }
    return s;
}

// Coarse FSM of Step 1 on U[0..N] (spacing H, r sampled at X_i), Gamma nodes
// fixed.  One warp.
template <class T>
struct FsmNode {
    T old, rh;
};
template <class T>
__device__ long long coarse_fsm(const DD1Args<T> &A, T *U, const T *rHc, const uint8_t *cfix, bool &conv) {
    auto load = [&](int j, FsmNode<T> &x) {
        x.old = U[j];
        x.rh = (cfix[j] != 0) | !finite_(rHc[j]) ? Num<T>::nan() : rHc[j];
    };
    auto f = [](const FsmNode<T> &x, T b, T a) { return fsm_chain(fsm_rest(x.old, x.rh, a), x.rh, b); };
    auto link = [](const FsmNode<T> &x, T b) { return Num<T>::add(b, x.rh); };
    return coarse_sweeps<T, FsmNode<T>>(A, U, load, link, f, f, conv);
}

// Step 4: weighted Gauss-Seidel sweeps of Un; ONE: theta = 1.  One warp.
template <class T>
struct WeightNode {
    T old, rH, uk, cold;
    int w;       // the only wind at which the weighted value is taken, 2 for none
    bool fixed;
};
template <bool ONE, class T>
__device__ long long weighted_sweeps(const DD1Args<T> &A, T *Un, const T *uk, const T *Cold, const T *rHc,
                                     const int8_t *W, const int8_t *wk, const uint8_t *cfix, bool &conv) {
    const T inf = Num<T>::inf(), theta = A.theta;
    auto load = [&](int j, WeightNode<T> &x) {
        x.old = Un[j];
        x.rH = rHc[j];
        x.uk = uk[j];
        x.cold = Cold[j];
        x.w = (W[j] == wk[j]) & Num<T>::lt(x.cold, inf) ? W[j] : 2;
        x.fixed = cfix[j] != 0;
    };
    // both neighbours' weighted values, so that the chain has no comparison in it
    auto weighted = [&](const WeightNode<T> &x, T Ut) {
        const T d = Num<T>::sub(Ut, x.cold);
        return Num<T>::add(x.uk, ONE ? d : Num<T>::mul(theta, d));
    };
    auto pick = [&](const WeightNode<T> &x, T behind, T ahead, bool by_ahead, int Wt) {
        const T ua = Num<T>::add(ahead, x.rH), ub = Num<T>::add(behind, x.rH);
        const T va = weighted(x, ua), vb = weighted(x, ub);
        const bool take = (Wt == x.w) & Num<T>::lt(by_ahead ? ua : ub, inf);
        const T v = take ? (by_ahead ? va : vb) : x.uk;
        return x.fixed ? x.old : v;
    };
    auto down = [&](const WeightNode<T> &x, T behind, T ahead) {
        const bool left = Num<T>::lt(ahead, behind);
        return pick(x, behind, ahead, left, left ? 1 : -1);
    };
    auto up = [&](const WeightNode<T> &x, T behind, T ahead) {
        const bool left = Num<T>::lt(behind, ahead);
        return pick(x, behind, ahead, !left, left ? 1 : -1);
    };
    auto link = [&](const WeightNode<T> &x, T behind) { return weighted(x, Num<T>::add(behind, x.rH)); };
    return coarse_sweeps<T, WeightNode<T>>(A, Un, load, link, down, up, conv);
}

// Causal sweep in both directions until nothing changes (values only rise to a
// neighbour's, so it ends; the cap is a guard); the rounds run.  One warp.
template <class T>
struct CausalNode {
    T old;
    int w;
};
template <class T>
__device__ int causal_rounds(int N, T *Un, const int8_t *W) {
    const T inf = Num<T>::inf();
    auto load = [&](int j, CausalNode<T> &x) {
        x.old = Un[j];
        x.w = W[j];
    };
    auto rise = [&](const CausalNode<T> &x, T behind, int w) {
        return (x.w == w) & Num<T>::lt(x.old, behind) & Num<T>::lt(behind, inf) ? behind : x.old;
    };
    auto up = [&](const CausalNode<T> &x, T behind, T) { return rise(x, behind, 1); };
    auto down = [&](const CausalNode<T> &x, T behind, T) { return rise(x, behind, -1); };
    auto link = [](const CausalNode<T> &, T behind) { return behind; };
    const long long round_cap = (long long)(N + 2) * (N + 2);
    int rounds = 0;
    bool changed;
    do {
        ++rounds;
        changed = coarse_sweep<1, T, CausalNode<T>>(N + 1, Un, load, link, up);
        changed = coarse_sweep<-1, T, CausalNode<T>>(N + 1, Un, load, link, down) || changed;
    } while (changed && rounds < round_cap);
    return rounds;
}

// A subinterval where its sweeps read and write it.  SM: u and r h (NaN where
// fsm_chain wants it) of its M + 1 nodes and one that stays after them in shared
// memory; else the interior of u, r and Gamma in global memory and the ends, which
// two subintervals share, in `ends`.
template <class T, bool SM>
struct Line {
    using I = std::conditional_t<SM, int, long long>;
    T *u, *ends;
    const T *rh;  // r in global memory
    const uint8_t *gm;
    T h;
    I M;
    __device__ __forceinline__ T *slot(I j) const { return SM || (j > 0 && j < M) ? u + j : ends + (j == 0 ? 0 : 1); }
    __device__ __forceinline__ T rh_at(I j) const {
        if (SM) return rh[j];
        const T v = Num<T>::mul(rh[j], h);
        return (gm[j] != 0) | !finite_(v) ? Num<T>::nan() : v;
    }
    // position p of a sweep in direction DIR; +inf past the end
    template <int DIR>
    __device__ __forceinline__ void read(I p, bool on, T &old, T &rh) const {
        const I j = DIR > 0 ? p : M - p;
        const bool in = on && p <= M;
        if (SM) {
            const I k = in ? j : M + 1;
            old = u[k];
            rh = this->rh[k];
        } else {
            old = Num<T>::inf();
            rh = Num<T>::nan();
            if (in) {
                old = *slot(j);
                rh = rh_at(j);
            }
        }
    }
};

// One sweep of a subinterval in direction DIR by DD1_G neighbouring lanes;
// returns whether this lane changed a value.  All lanes of the warp take part;
// groups without work (on = false) change nothing.  DD1_S x DD1_G positions are
// checked at once.  Where they change, all lanes add up the chain alike as if
// every node but the first followed its predecessor (one addition a node); each
// then compares its own, and only if one did not follow are they walked with the
// comparisons in the chain.
constexpr int DD1_S = 4;

template <int DIR, class T, bool SM>
__device__ __forceinline__ bool sub_sweep(const Line<T, SM> &L, bool on) {
    using I = typename Line<T, SM>::I;
    constexpr int G = DD1_G, S = DD1_S;
    const int lane = threadIdx.x & (G - 1);
    T carry = Num<T>::inf();
    bool ch = false;
#pragma unroll 1
    for (I p0 = 0; p0 <= L.M; p0 += S * G) {
        T old[S], rh[S], rest[S], v[S], over, unused;
#pragma unroll
        for (int i = 0; i < S; ++i) L.template read<DIR>(p0 + i * G + lane, on, old[i], rh[i]);
        L.template read<DIR>(p0 + S * G, on, over, unused);
        bool moved = false;
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const T first = i + 1 < S ? __shfl_sync(FULL, old[i + 1 < S ? i + 1 : i], 0, G) : over;
            T ahead = __shfl_down_sync(FULL, old[i], 1, G);
            if (lane == G - 1) ahead = first;
            const T last = i > 0 ? __shfl_sync(FULL, old[i > 0 ? i - 1 : 0], G - 1, G) : carry;
            T behind = __shfl_up_sync(FULL, old[i], 1, G);
            if (lane == 0) behind = last;
            rest[i] = fsm_rest(old[i], rh[i], ahead);
            moved |= !same_bits(fsm_chain(rest[i], rh[i], behind), old[i]);
        }
        if (!__any_sync(FULL, moved)) {
            carry = __shfl_sync(FULL, old[S - 1], G - 1, G);
            continue;
        }
        const bool kept = !group_any(moved);  // this group's are done
        const int left = (int)min((I)(S * G), L.M + 1 - p0);  // positions of the line here
        T t = fsm_chain(__shfl_sync(FULL, rest[0], 0, G), __shfl_sync(FULL, rh[0], 0, G), carry);
        bool followed = true;
#pragma unroll
        for (int i = 0; i < S; ++i) {
            v[i] = t;
            if (i * G < left) {
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    if (i + k > 0) t = Num<T>::add(t, __shfl_sync(FULL, rh[i], k, G));
                    if (lane == k) v[i] = t;
                }
                followed &= (i == 0 && lane == 0) | (i * G + lane >= left) | Num<T>::below(v[i], rest[i]);
            }
        }
        if (__any_sync(FULL, !kept && !followed)) {
            t = carry;
#pragma unroll
            for (int i = 0; i < S; ++i) {
#pragma unroll 1
                for (int k = 0; k < min(G, left - i * G); ++k) {
                    t = fsm_chain(__shfl_sync(FULL, rest[i], k, G), __shfl_sync(FULL, rh[i], k, G), t);
                    if (lane == k) v[i] = t;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const I p = p0 + i * G + lane;
            if (kept) v[i] = old[i];
            if (on && p <= L.M && !same_bits(v[i], old[i])) {
                ch = true;
                *L.slot(DIR > 0 ? p : L.M - p) = v[i];
            }
        }
        carry = __shfl_sync(FULL, v[S - 1], G - 1, G);
    }
    __syncwarp();
    return ch;
}

// Steps 2-3 on subinterval `sub` by a group of DD1_G lanes, given U and W at its
// two ends; all lanes of the warp call it, on = false for groups without one.
// Step 2: a Gamma node is fixed at g; an end where the coarse wind points into
// the subinterval (W = +1 at its left end, W = -1 at its right end) starts at
// U, every other node at +inf.  Step 3: FSM sweeps (right-to-left first) until
// one changes nothing or the cap is reached.  The values are left in L; the ends'
// values, winds and echo flags go to the end-copy arrays.
// Returns the sweeps run; conv = false if the cap stopped them.
template <class T, bool SM>
__device__ long long solve_sub(const DD1Args<T> &A, const Line<T, SM> &L, int sub, bool on, T Ul, T Ur, int Wl, int Wr,
                               bool &conv) {
    const T inf = Num<T>::inf();
    const long long M = A.M, f0 = (long long)sub * M;
    const int lane = threadIdx.x & (DD1_G - 1);
    const uint8_t *gm = A.gamma + f0;
    const T *g = A.g + f0;
    const bool fix0 = gm[0] != 0, fixM = gm[M] != 0;
    const bool in0 = !fix0 && Wl > 0, inM = !fixM && Wr < 0;
    const T s0 = fix0 ? gamma_value(g[0]) : (in0 ? Ul : inf);
    const T sM = fixM ? gamma_value(g[M]) : (inM ? Ur : inf);
    if (on) {
        for (long long j0 = 1 + lane; j0 < M; j0 += 8 * DD1_G) {
            uint8_t f[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) f[i] = j0 + i * DD1_G < M ? gm[j0 + i * DD1_G] : 0;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (j0 + i * DD1_G < M) L.u[j0 + i * DD1_G] = f[i] ? gamma_value(g[j0 + i * DD1_G]) : inf;
        }
        if (lane == 0) {
            *L.slot(0) = s0;
            *L.slot(M) = sM;
        }
    }
    __syncwarp();
    long long s = 0, done = 0;  // sweeps of the warp, of this group
    conv = false;
    bool go = on;
    while (s < A.max_fsm && __any_sync(FULL, go)) {
        const bool ch = group_any((s % 2 == 0) ? sub_sweep<-1>(L, go) : sub_sweep<1>(L, go));
        ++s;
        if (go) {
            done = s;
            if (!ch) {
                conv = true;
                go = false;
            }
        }
    }
    if (!on || lane != 0) return done;
    // winds of the ends at the final values (0 at Gamma and at +inf)
    const T *r = A.r + f0;
    const T e0 = *L.slot(0), eM = *L.slot(M);
    int w0 = 0, wM = 0;
    if (!fix0 && e0 < inf) (void)ch1(inf, *L.slot(1), Num<T>::mul(r[0], A.h), w0);
    if (!fixM && eM < inf) (void)ch1(*L.slot(M - 1), inf, Num<T>::mul(r[M], A.h), wM);
    const bool echo0 = in0 && e0 == s0, echoM = inM && eM == sM;
    if (echo0) w0 = Wl;
    if (echoM) wM = Wr;
    A.geu[2 * sub] = e0;
    A.geu[2 * sub + 1] = eM;
    A.gew[2 * sub] = (int8_t)w0;
    A.gew[2 * sub + 1] = (int8_t)wM;
    A.gee[2 * sub] = echo0 ? 1 : 0;
    A.gee[2 * sub + 1] = echoM ? 1 : 0;
    return done;
}

template <class T, bool SM>
__global__ void __launch_bounds__(DD1_THREADS, 1) k_dd1(DD1Args<T> A) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int N = A.N;
    const long long M = A.M;
    const T inf = Num<T>::inf();
    const long long lim = spin_limit();
    DD1Ctl *ctl = A.ctl;
    const int tid = threadIdx.x, nt = blockDim.x;
    const bool lead = blockIdx.x == 0;
    // CTA 0's coarse state
    T *U = reinterpret_cast<T *>(smem);
    T *Un = U + (N + 1);     // the U being built by Step 4
    T *uk = Un + (N + 1);    // u^k of Step 3's choice
    T *Cold = uk + (N + 1);  // C_H(U^k)
    T *rHc = Cold + (N + 1); // r(X_i) H
    int8_t *W = reinterpret_cast<int8_t *>(rHc + (N + 1));
    int8_t *wk = W + (N + 1);
    uint8_t *cfix = reinterpret_cast<uint8_t *>(wk + (N + 1));
    __shared__ unsigned long long s_coarse_upd, s_coarse_max, s_coarse_caps;
    __shared__ int s_causal_max;
    __shared__ T s_delta;

    if (lead) {
        if (tid == 0) {
            s_coarse_upd = s_coarse_max = s_coarse_caps = 0;
            s_causal_max = 0;
            s_delta = inf;
            ctl->fsm_max = ctl->fsm_caps = ctl->fine_upd = 0;
        }
        for (int i = tid; i <= N; i += nt) {
            const long long f = (long long)i * M;
            cfix[i] = A.gamma[f] ? 1 : 0;
            U[i] = A.gamma[f] ? gamma_value(A.g[f]) : inf;
            rHc[i] = Num<T>::mul(A.r[f], A.H);
        }
        __syncthreads();
        // Step 1: FSM on the coarse grid, then the winds W^0
        if (tid < 32) {
            bool conv;
            const long long s = coarse_fsm(A, U, rHc, cfix, conv);
            if (tid == 0) {
                s_coarse_max = (unsigned long long)s;
                s_coarse_caps = conv ? 0 : 1;
                s_coarse_upd = (unsigned long long)s * (N + 1);
            }
        }
        __syncthreads();
        for (int i = tid; i <= N; i += nt) {
            int w = 0;
            if (!cfix[i] && U[i] < inf) (void)ch1_at(U, i, N, rHc[i], w);
            W[i] = (int8_t)w;
            A.gU[i] = U[i];
            A.gW[i] = (int8_t)w;
        }
    }
    bool ok = grid_barrier(ctl->bar, &ctl->err, lim);
    int k = 0, converged = 0;
    const int grp = tid / DD1_G, sub = blockIdx.x * A.per + grp;
    const bool mine = grp < A.per && sub < N, group = (tid & ~31) / DD1_G < A.per;
    __shared__ T s_ends[2 * (DD1_THREADS / DD1_G)];
    Line<T, SM> L;
    L.M = (typename Line<T, SM>::I)M;
    L.h = A.h;
    L.ends = s_ends + 2 * grp;
    L.gm = A.gamma + (mine ? (long long)sub * M : 0);
    if (SM) {
        const long long pitch = dd1_pitch(M);
        // (groups past the last one only read the node after its nodes)
        T *const rh = reinterpret_cast<T *>(smem + dd1_coarse_bytes<T>(N)) + (size_t)2 * min(grp, A.per - 1) * pitch;
        L.u = rh + pitch;
        L.rh = rh;
        Line<T, false> G;  // r h as the other form reads it
        G.rh = A.r + (mine ? (long long)sub * M : 0);
        G.gm = L.gm;
        G.h = A.h;
        if (mine) {
#pragma unroll 4
            for (long long j = tid % DD1_G; j <= M; j += DD1_G) rh[j] = G.rh_at(j);
        }
        if (grp < A.per) {
            rh[M + 1] = Num<T>::nan();
            L.u[M + 1] = inf;
        }
        __syncthreads();
    } else {
        L.u = A.u + (mine ? (long long)sub * M : 0);
        L.rh = A.r + (mine ? (long long)sub * M : 0);
    }
    while (ok) {
        // Steps 2-3: every subinterval on its own (U, W written by another SM:
        // read past L1)
        if (group) {
            bool cv;
            const int at = mine ? sub : 0;
            const long long s = solve_sub(A, L, at, mine, __ldcg(A.gU + at), __ldcg(A.gU + at + 1), (int)__ldcg(A.gW + at),
                                          (int)__ldcg(A.gW + at + 1), cv);
            if (mine && tid % DD1_G == 0) {
                atomicMax(&ctl->fsm_max, (unsigned long long)s);
                if (!cv) atomicAdd(&ctl->fsm_caps, 1ull);
                atomicAdd(&ctl->fine_upd, (unsigned long long)s * (unsigned long long)(M + 1));
            }
        }
        if (!(ok = grid_barrier(ctl->bar, &ctl->err, lim))) break;
        if (lead) {
            // Step 3's choice of u^k_i and w^k_i between the two fine copies
            for (int i = tid; i <= N; i += nt) {
                if (i == 0) {
                    uk[0] = __ldcg(A.geu);
                    wk[0] = __ldcg(A.gew);
                } else if (i == N) {
                    uk[N] = __ldcg(A.geu + 2 * N - 1);
                    wk[N] = __ldcg(A.gew + 2 * N - 1);
                } else {
                    const T uL = __ldcg(A.geu + 2 * i - 1), uR = __ldcg(A.geu + 2 * i);
                    const int wL = __ldcg(A.gew + 2 * i - 1), wR = __ldcg(A.gew + 2 * i);
                    const int eL = __ldcg(A.gee + 2 * i - 1), eR = __ldcg(A.gee + 2 * i);
                    bool takeL;
                    if (wL == 1 && wR == 1) takeL = true;          // wind from left to right
                    else if (wL == -1 && wR == -1) takeL = false;  // wind from right to left
                    else if (eL != eR) takeL = eR != 0;            // the computed copy of the two
                    else takeL = !(uR < uL);                       // minimum, a tie to the left copy
                    uk[i] = takeL ? uL : uR;
                    wk[i] = (int8_t)(takeL ? wL : wR);
                }
            }
            __syncthreads();
            int stop = 0;
            if (k == A.max_iter) stop = 1;
            else if (k >= 1 && s_delta < A.tol) stop = 2;
            if (!stop) {
                // Step 4: C_H(U^k), then weighted Gauss-Seidel sweeps from the
                // FSM initialisation
                for (int i = tid; i <= N; i += nt) {
                    int w;
                    Cold[i] = ch1_at(U, i, N, rHc[i], w);
                    Un[i] = cfix[i] ? gamma_value(A.g[(long long)i * M]) : inf;
                }
                __syncthreads();
                if (tid < 32) {
                    bool conv;
                    const long long s = A.theta == T(1)
                                            ? weighted_sweeps<true>(A, Un, uk, Cold, rHc, W, wk, cfix, conv)
                                            : weighted_sweeps<false>(A, Un, uk, Cold, rHc, W, wk, cfix, conv);
                    for (int i = tid; i <= N; i += 32) W[i] = wk[i];
                    __syncwarp();
                    const int rounds = causal_rounds(N, Un, W);
                    T d = T(0);
#pragma unroll 4
                    for (int i = tid; i <= N; i += 32)
                        if (!(Un[i] == U[i])) {
                            const T t = abs_(Num<T>::sub(Un[i], U[i]));
                            if (t > d) d = t;
                        }
                    for (int m = 16; m; m >>= 1) {
                        const T t = __shfl_xor_sync(FULL, d, m);
                        if (t > d) d = t;
                    }
                    if (tid == 0) {
                        if (!conv) ++s_coarse_caps;
                        if ((unsigned long long)s > s_coarse_max) s_coarse_max = (unsigned long long)s;
                        s_coarse_upd += (unsigned long long)s * (N + 1);
                        if (rounds > s_causal_max) s_causal_max = rounds;
                        s_delta = d;
                    }
                }
                __syncthreads();
                T *t = U;  // U^{k+1} is the U just built
                U = Un;
                Un = t;
                for (int i = tid; i <= N; i += nt) {
                    A.gU[i] = U[i];
                    A.gW[i] = W[i];
                }
            }
            if (tid == 0) ctl->stop = stop;
        }
        if (!(ok = grid_barrier(ctl->bar, &ctl->err, lim))) break;
        const int stop = *(volatile int *)&ctl->stop;
        if (stop) {
            converged = stop == 2 ? 1 : 0;
            break;
        }
        ++k;
    }
    if (SM && ok && mine)
        for (long long j = 1 + tid % DD1_G; j < M; j += DD1_G) A.u[(long long)sub * M + j] = L.u[j];
    if (!lead) return;
    // the patched fine solution: coarse nodes take u^k
    if (ok)
        for (int i = tid; i <= N; i += nt) A.u[(long long)i * M] = uk[i];
    if (tid == 0 && A.stats) {
        eik_dd_stats *o = A.stats;
        o->iters = k;
        o->converged = converged;
        o->error = *(volatile int *)&ctl->err;
        o->causal_rounds_max = s_causal_max;
        o->fsm_sweeps_max = (int64_t)*(volatile unsigned long long *)&ctl->fsm_max;
        o->coarse_sweeps_max = (int64_t)s_coarse_max;
        o->fsm_cap_hits = (int64_t)*(volatile unsigned long long *)&ctl->fsm_caps;
        o->coarse_cap_hits = (int64_t)s_coarse_caps;
        o->last_delta = k >= 1 ? (double)s_delta : INFINITY;
        o->fine_updates = (int64_t)*(volatile unsigned long long *)&ctl->fine_upd;
        o->coarse_updates = (int64_t)s_coarse_upd;
        o->launches = 1;
        o->fine_solves_skipped = 0;
    }
}

// --------------------------------------------------------------------------
// Host side
// --------------------------------------------------------------------------
bool dd1_validate(const eik_grid *grid, const eik_dd_params *p) {
    if (!valid_grid_common(grid, 1)) return false;
    const long long n = grid->n[0];
    const int N = p->tiles[0];
    if (N < 1 || (n - 1) % N != 0) {
        set_error("tiles[0] = %d does not divide n[0]-1 = %lld", N, n - 1);
        return false;
    }
    if (N > DD1_MAX_SUB) {
        set_error("1-D solve: %d subintervals, at most %d (the coarse state is held in shared memory)", N,
                  DD1_MAX_SUB);
        return false;
    }
    const long long M = (n - 1) / N;
    if (p->coarse_ratio != M) {
        set_error("1-D solve: the coarse nodes are the subinterval ends, so coarse_ratio must be (n-1)/tiles[0] = %lld",
                  M);
        return false;
    }
    if (p->max_iter < 0 || p->max_iter > 100000 || p->max_fsm_sweeps < 1 || p->max_coarse_sweeps < 1 ||
        p->max_fsm_sweeps > MAX_SWEEPS || p->max_coarse_sweeps > MAX_SWEEPS) {
        set_error("max_iter must be in [0, 100000] and sweep caps in [1, %lld]", MAX_SWEEPS);
        return false;
    }
    if (!std::isfinite(p->theta) || std::isnan(p->tol)) {
        set_error("theta must be finite and tol a number");
        return false;
    }
    if (p->theta_adaptive) {
        set_error("the per-node weight of Sec. 4.2 is built for the 2-D and 3-D solves only");
        return false;
    }
    return true;
}

size_t dd1_workspace_size(const eik_grid *grid, const eik_dd_params *p) {
    return grid->dtype == EIK_F64 ? dd1_ws_bytes<double>(p->tiles[0]) : dd1_ws_bytes<float>(p->tiles[0]);
}

template <class T>
static int dd1_run_t(const eik_grid *grid, const void *r, const uint8_t *gamma, const void *g,
                     const eik_dd_params *p, void *u_out, void *ws, eik_dd_stats *stats, cudaStream_t s) {
    DD1Args<T> A;
    memset(&A, 0, sizeof(A));
    A.r = static_cast<const T *>(r);
    A.gamma = gamma;
    A.g = static_cast<const T *>(g);
    A.u = static_cast<T *>(u_out);
    A.stats = stats;
    A.N = p->tiles[0];
    A.M = (grid->n[0] - 1) / A.N;
    A.h = (T)grid->h;
    A.H = (T)((double)A.M * grid->h);
    A.theta = (T)p->theta;
    A.tol = (T)p->tol;
    A.max_iter = p->max_iter;
    A.max_fsm = p->max_fsm_sweeps;
    A.max_coarse = p->max_coarse_sweeps;
    const int N = A.N;
    char *w = static_cast<char *>(ws);
    A.ctl = reinterpret_cast<DD1Ctl *>(w);
    w += al256(sizeof(DD1Ctl));
    A.gU = reinterpret_cast<T *>(w);
    w += al256((size_t)(N + 1) * sizeof(T));
    A.gW = reinterpret_cast<int8_t *>(w);
    w += al256((size_t)(N + 1));
    A.geu = reinterpret_cast<T *>(w);
    w += al256((size_t)2 * N * sizeof(T));
    A.gew = reinterpret_cast<int8_t *>(w);
    w += al256((size_t)2 * N);
    A.gee = reinterpret_cast<uint8_t *>(w);

    size_t smem = dd1_coarse_bytes<T>(N);
    int rc, dev, nsm = 0, optin = 0, coop = 0;
    if ((rc = cuda_check(cudaGetDevice(&dev), "cudaGetDevice"))) return rc;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if ((long long)smem > optin || !coop) {
        set_error("1-D solve needs %zu bytes of shared memory (limit %d) and cooperative launch", smem, optin);
        return EIK_EUNSUPPORTED;
    }
    // subintervals spread over one CTA per SM, DD1_G lanes each, in shared memory
    // where they fit (1024 of 1001 FP64 nodes: 1.17 ms a solve, in global memory 1.49 ms)
    A.per = (N + nsm - 1) / nsm;
    const int nblk = (N + A.per - 1) / A.per;
    const int threads = std::max(32, (A.per * DD1_G + 31) / 32 * 32);
    const double lines = 2.0 * A.per * (double)dd1_pitch(A.M) * sizeof(T);
    const bool in_smem = smem + lines + 2048 <= optin;
    if (in_smem) smem += (size_t)lines;
    void (*const kernel)(DD1Args<T>) = in_smem ? k_dd1<T, true> : k_dd1<T, false>;
    if ((rc = cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "attr")))
        return rc;
    int per_sm = 0;
    if ((rc = cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem), "occ")))
        return rc;
    if (per_sm * nsm < nblk) {
        set_error("1-D solve needs %d co-resident CTAs, the device holds %d", nblk, per_sm * nsm);
        return EIK_EUNSUPPORTED;
    }
    if ((rc = cuda_check(cudaMemsetAsync(A.ctl, 0, sizeof(DD1Ctl), s), "clear control words"))) return rc;
    void *args[] = {&A};
    const int tok = prof_begin("dd1_iteration", s);
    rc = cuda_check(cudaLaunchCooperativeKernel((void *)kernel, nblk, threads, args, smem, s), "dd1 launch");
    prof_end(tok, s);
    return rc;
}

int dd1_run(const eik_grid *grid, const void *r, const uint8_t *gamma, const void *g, const eik_dd_params *p,
            void *u_out, void *ws, eik_dd_stats *stats, cudaStream_t s) {
    if (grid->dtype == EIK_F64) return dd1_run_t<double>(grid, r, gamma, g, p, u_out, ws, stats, s);
    return dd1_run_t<float>(grid, r, gamma, g, p, u_out, ws, stats, s);
}

}  // namespace eik
