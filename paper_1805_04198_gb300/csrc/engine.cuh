// engine.cuh -- warp-systolic Gauss-Seidel sweep engine for one 2-D grid box.
//
// A sweep of the fast sweeping method (Sec. 1.1) visits the nodes in one of
// the 2^d orderings; node (x, y) then reads its upwind-in-the-ordering
// neighbours already updated in this sweep and the other two from before it.
// Any schedule that respects exactly those four dependencies gives the same
// result as the serial loop nest.  The schedule used here:
//
//  * the box is cut into 32-column blocks; warp w owns physical block w for the
//    whole run, lane l one column of it (lane order follows the sweep sign of
//    x, so lane 0 is the upwind side);
//  * at step s lane l updates logical row s - l: its left neighbour (new) comes
//    from lane l-1 by a register shuffle, its upper neighbour (new) is the
//    value it produced one step earlier, its right neighbour (old) is lane
//    l+1's prefetched lower neighbour, shuffled down;
//  * the block's rows stream through a 64-row shared-memory ring in chunks of
//    8 rows, copied from global memory by cp.async three chunks ahead and
//    written back as soon as all 32 lanes finished them.  A row's ring slot is
//    its physical index mod 64 and the sign of y alternates from sweep to
//    sweep, so the first 64 rows of a sweep are still in the ring from the one
//    before and are not read again;
//  * the block's last lane hands its new column to the next block's warp
//    through a column buffer whose unwritten elements hold a reserved NaN: the
//    value is its own flag, so no fence and no flag word sit on the hand-off
//    path, and the reader puts the NaN back.  It reads the next block's first
//    column (old values) from global memory, one chunk ahead;
//  * per-node read-only data ("statics") are stored pre-skewed per sweep
//    direction, 16 bytes (consecutive steps) of a lane together, and go through
//    a small shared ring, so a chunk of one static is two 16-byte copies and two
//    16-byte reads per lane (FP32);
//  * positions outside the box hold neutral values (P::pad() in the state, the
//    policy's inert static), so columns need no tests; rows are tested only in
//    the chunks that touch the ends of the box;
//  * there is no CTA-wide barrier between sweeps: a warp starts sweep k+1 as
//    soon as its own block and the block whose old column it reads have
//    finished sweep k, so the pipeline reverses direction without draining
//    when the x sign flips.  A sweep that changes no node anywhere marks a
//    fixed point; the engine then stops (sweeps a warp had already begun
//    speculatively change nothing).
//
// What bounds it: the chain of one step (shuffle, two differences, square
// root, select, minimum), NX + NY of them per sweep, not memory; two boxes of
// nine warps on an SM issue in two of three cycles.  257^2 FP32 in one CTA 51 us
// a sweep (85 with flags and fences, re-read rows and tests in the step), FP64 308
// us; a full 4097^2 FP32 grid 0.97 ms a sweep (2.06).  The sweep direction is a
// run-time value (one copy of the step code for all four orderings); policies that
// do not distinguish the sides of an axis (P::SYM) are given the two axis minima.
//
// Storage of the state u: strip-major [block][row][32] (row = physical y,
// 32 = physical x within the block), padded to a whole number of blocks with
// P::pad().  One-sided differences at the box edges come for free: missing
// neighbours are +inf.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace eik {

constexpr int CH = 8;             // rows (and steps) per chunk
constexpr int RROWS = 64;         // u ring rows per warp (power of two)
constexpr int SRCH = 3;           // statics chunks held in the statics ring
constexpr int LEAD = 3;           // u chunks copied ahead of the current one
constexpr int MAX_BOX_ROWS = (1 << 13) - 1;
constexpr long long MAX_SWEEPS = 1ll << 17;

__host__ __device__ inline int ceil32(int v) { return (v + 31) >> 5; }

// Element index of node (i, j) of a strip-major box of height my.
__host__ __device__ inline size_t box_index(int i, int j, int my) {
    return ((size_t)(i >> 5) * my + j) * 32 + (i & 31);
}

// Steps of one statics stream, padded to whole chunks plus at least the lead (two
// chunks ahead of the last).  Plain sweeping and the adjoint take a chunk less than
// the decomposition: that makes room for their hand-off columns in the workspace
// sizes that callers know.
__host__ __device__ inline int nstep_padded(int ny) { return ((ny + 31 + CH - 1) / CH) * CH + 4 * CH; }
__host__ __device__ inline int nstep_whole_grid(int ny) { return nstep_padded(ny) - CH; }

// Sweep direction d in [0, 4): bit 1 = sign of x, bit 0 = sign of y (set =
// +1).  The paper's loop nest (x sign outermost, -1 first) visits d = 0..3 in
// order, so sweep k uses d = k % 4.
__host__ __device__ inline int dir_sx(int d) { return (d & 2) ? 1 : -1; }
__host__ __device__ inline int dir_sy(int d) { return (d & 1) ? 1 : -1; }

// Skewed statics: one stream of nstepp x 32 elements per direction and logical
// block.  What lane l reads at step s is element skew_off<T>(s, l): within a
// chunk of 8 steps, 16 bytes of consecutive steps of a lane, the 32 lanes side
// by side, so that a chunk is read with 16-byte accesses of whole 512-byte rows.
template <class T>
__host__ __device__ inline size_t skew_off(int s, int l) {
    constexpr int E = sizeof(T) == 1 ? CH : 16 / (int)sizeof(T);
    return ((size_t)(s / E) * 32 + l) * E + s % E;
}
// Its inverse.
template <class T>
__host__ __device__ inline void skew_pos(unsigned e, int &s, int &l) {
    constexpr unsigned E = sizeof(T) == 1 ? CH : 16 / (int)sizeof(T);
    s = (int)(e / (32 * E) * E + e % E);
    l = (int)(e / E % 32);
}

// Index of node (i, j) of a box (width -> nb blocks, height my) in the skewed
// statics: [direction][logical block][stream].
template <class T>
__host__ __device__ inline size_t skew_index(int d, int i, int j, int nb, int my, int nstepp) {
    int sx = dir_sx(d), sy = dir_sy(d);
    int b = i >> 5, pc = i & 31;
    int q = sx > 0 ? b : nb - 1 - b;
    int l = sx > 0 ? pc : 31 - pc;
    int lr = sy > 0 ? j : my - 1 - j;
    return ((size_t)d * nb + q) * nstepp * 32 + skew_off<T>(lr + l, l);
}

// Inverse of skew_index for kernels that write the statics in storage order:
// element e -> node (x, y); false where the position is outside the box.
template <class T>
__device__ __forceinline__ bool skew_node(size_t e, int nx, int my, int nb, int nstepp, int &x, int &y) {
    const unsigned stream = (unsigned)nstepp * 32;
    const unsigned dq = (unsigned)(e / stream);
    int s, l;
    skew_pos<T>((unsigned)(e - (size_t)dq * stream), s, l);
    const int q = (int)(dq % nb), d = (int)(dq / nb);
    const bool px = dir_sx(d) > 0;
    x = 32 * (px ? q : nb - 1 - q) + (px ? l : 31 - l);
    const int lr = s - l;
    y = dir_sy(d) > 0 ? lr : my - 1 - lr;
    return x < nx && lr >= 0 && lr < my;
}

// Packs NCH channels of a field into skewed statics (out + c * chan), positions
// outside the box get `pad`; get(c, x, y) is the value at a node.  A stream reads
// the field along diagonals, 32 rows for 32 neighbouring columns: gathered from
// global memory that is a transaction per element (5 channels of 64 fields of
// 1025^2: 4.3 ms, one L1 wavefront an element).  So rows are loaded as rows into a
// tile of one block's 32 columns and read diagonally there, where the lanes of a
// warp stand in different banks (2.2 ms).  A tile serves 64 steps of all four
// directions: those whose group of steps starts at its row, counted from the
// bottom or from the top, and the 31 rows before and after that they reach.
constexpr int PACK_ROWS = 64;
template <class T, int NCH, class Get>
__device__ __forceinline__ void skew_pack(T *out, size_t chan, int nx, int my, int nb, int nstepp, size_t bid,
                                          size_t nbid, T pad, Get get) {
    constexpr int E = 16 / (int)sizeof(T), LE = sizeof(T) == 4 ? 2 : 1, S = PACK_ROWS, R = S + 62;
    __shared__ T tile[R * 32];
    const int wmin = my - nstepp, nwin = (nstepp - wmin + S - 1) / S, ng = nstepp >> LE;
    const int lane = threadIdx.x & 31;
    for (size_t t = bid; t < (size_t)nb * nwin * NCH; t += nbid) {
        const int c = (int)(t % NCH), u = (int)(t / NCH), b = u / nwin, w0 = wmin + (u - b * nwin) * S;
        __syncthreads();
        for (int e = threadIdx.x; e < R * 32; e += blockDim.x) {
            const int y = w0 - 31 + (e >> 5), x = 32 * b + lane;
            tile[e] = x < nx && y >= 0 && y < my ? get(c, x, y) : pad;
        }
        __syncthreads();
#pragma unroll
        for (int sy = 0; sy < 2; ++sy) {
            // groups of E steps whose first step s0 has s0 (sy = 1) or my - 1 - s0 in [w0, w0 + S)
            const int lo = max(0, sy ? (w0 + E - 1) >> LE : ((my - 1 - w0 - S) >> LE) + 1);
            const int hi = min(ng, sy ? (w0 + S + E - 1) >> LE : ((my - 1 - w0) >> LE) + 1);
            for (int k = threadIdx.x >> 5; k < 2 * (hi - lo); k += blockDim.x >> 5) {
                const int px = k & 1, gq = lo + (k >> 1), col = px ? lane : 31 - lane;
                union { T v[E]; uint4 w; } o;
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    const int lr = E * gq + i - lane, y = sy ? lr : my - 1 - lr;
                    o.v[i] = tile[(y - w0 + 31) * 32 + col];
                }
                const size_t stream = (size_t)(2 * px + sy) * nb + (px ? b : nb - 1 - b);
                reinterpret_cast<uint4 *>(out + c * chan + stream * nstepp * 32)[gq * 32 + lane] = o.w;
            }
        }
    }
}

template <class T, int NST>
struct Box {
    T *u;                          // state, strip-major [nb][ny][32]
    const T *st[NST];              // skewed statics [4][nb][nstepp][32]
    const uint8_t *sb;             // skewed byte statics (may be null)
    int ny, nb, nstepp;
};

// Elements of one hand-off column.
__host__ __device__ inline size_t hand_elems(int ny) { return (size_t)((ny + CH - 1) / CH * CH); }

// Shared memory needed per CTA of `nw` warps (one warp per block).  With
// GLOBAL the hand-off columns and control words live in global memory.
template <class T, int NST, bool HASB, bool GLOBAL = false>
__host__ __device__ inline size_t engine_smem_bytes(int nw, int ny) {
    size_t per_warp = (size_t)RROWS * 32 * sizeof(T)                        // u ring
                      + (size_t)NST * SRCH * CH * 32 * sizeof(T)            // statics ring
                      + (size_t)2 * CH * sizeof(T)                          // halo of two chunks
                      + (GLOBAL ? 0 : hand_elems(ny) * sizeof(T))           // hand-off column
                      + (HASB ? (size_t)SRCH * CH * 32 : 0);                // byte statics ring
    return nw * per_warp + (GLOBAL ? 0 : (size_t)(32 + nw) * sizeof(int)) + 64;
}

// The shared memory by which a box is accepted or refused (EIK_EUNSUPPORTED):
// the documented size limit of subdomains and coarse grids, an upper bound of
// what the engine takes.
template <class T, int NST, bool HASB>
__host__ inline size_t engine_limit_bytes(int nw, int ny) {
    const size_t per_warp = (size_t)RROWS * 33 * sizeof(T) + (size_t)NST * SRCH * CH * 32 * sizeof(T) +
                            (size_t)((ny + 3) & ~3) * sizeof(T) + (HASB ? (size_t)SRCH * CH * 32 : 0);
    return nw * per_warp + (size_t)(32 + 2 * nw) * sizeof(int) + 64;
}

// Control words of a multi-CTA engine run (global memory, set by
// engine_global_init before the run): abort, stop_at, fin[8], chg[8], then
// done[nb].
__host__ __device__ inline size_t engine_global_ints(int nb) { return 32 + (size_t)nb; }

// Element access with the reserved NaN of the hand-off columns.
template <class T> struct Hand;
template <> struct Hand<float> {
    static __device__ __forceinline__ float empty() { return __uint_as_float(0x7fd5a5c3u); }
    static __device__ __forceinline__ bool is_empty(float v) { return __float_as_uint(v) == 0x7fd5a5c3u; }
};
template <> struct Hand<double> {
    static __device__ __forceinline__ double empty() { return __longlong_as_double(0x7ffad5a5c3b4e1f7ll); }
    static __device__ __forceinline__ bool is_empty(double v) {
        return __double_as_longlong(v) == 0x7ffad5a5c3b4e1f7ll;
    }
};

// 16 bytes of elements (shared memory by 32-bit address).
__device__ __forceinline__ void lds16(unsigned a, float *v) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds16(unsigned a, double *v) {
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a) : "memory");
}
// hand-off columns in shared memory: polled, so volatile
__device__ __forceinline__ void hand_lds16(unsigned a, float *v) {
    asm volatile("ld.volatile.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void hand_lds16(unsigned a, double *v) {
    asm volatile("ld.volatile.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a) : "memory");
}
__device__ __forceinline__ float lds1(unsigned a, float) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ double lds1(unsigned a, double) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts1(unsigned a, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void sts1(unsigned a, double v) {
    asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
// Predicated forms: a branch around one access costs more than the access.
#define EIK_PRED "{.reg .pred p; setp.ne.b32 p, %"
__device__ __forceinline__ void lds1_if(bool c, unsigned a, float &v) {
    asm volatile(EIK_PRED "2, 0; @p ld.shared.f32 %0, [%1];}" : "+f"(v) : "r"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void lds1_if(bool c, unsigned a, double &v) {
    asm volatile(EIK_PRED "2, 0; @p ld.shared.f64 %0, [%1];}" : "+d"(v) : "r"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void sts1_if(bool c, unsigned a, float v) {
    asm volatile(EIK_PRED "2, 0; @p st.shared.f32 [%0], %1;}" ::"r"(a), "f"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void sts1_if(bool c, unsigned a, double v) {
    asm volatile(EIK_PRED "2, 0; @p st.shared.f64 [%0], %1;}" ::"r"(a), "d"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void hand_sts_if(bool c, unsigned a, float v) {
    asm volatile(EIK_PRED "2, 0; @p st.volatile.shared.f32 [%0], %1;}" ::"r"(a), "f"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void hand_sts_if(bool c, unsigned a, double v) {
    asm volatile(EIK_PRED "2, 0; @p st.volatile.shared.f64 [%0], %1;}" ::"r"(a), "d"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void hand_stg_if(bool c, float *a, float v) {
    asm volatile(EIK_PRED "2, 0; @p st.volatile.global.f32 [%0], %1;}" ::"l"(a), "f"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void hand_stg_if(bool c, double *a, double v) {
    asm volatile(EIK_PRED "2, 0; @p st.volatile.global.f64 [%0], %1;}" ::"l"(a), "d"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void hand_ldg_if(bool c, const float *a, float &v) {
    asm volatile(EIK_PRED "2, 0; @p ld.volatile.global.f32 %0, [%1];}" : "+f"(v) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void hand_ldg_if(bool c, const double *a, double &v) {
    asm volatile(EIK_PRED "2, 0; @p ld.volatile.global.f64 %0, [%1];}" : "+d"(v) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void ldcg_if(bool c, const float *a, float &v) {
    asm volatile(EIK_PRED "2, 0; @p ld.global.cg.f32 %0, [%1];}" : "+f"(v) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void ldcg_if(bool c, const double *a, double &v) {
    asm volatile(EIK_PRED "2, 0; @p ld.global.cg.f64 %0, [%1];}" : "+d"(v) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void stcg16_if(bool c, void *a, const uint4 &v) {
    asm volatile(EIK_PRED "5, 0; @p st.global.cg.v4.u32 [%0], {%1, %2, %3, %4};}" ::"l"(a), "r"(v.x), "r"(v.y),
                 "r"(v.z), "r"(v.w), "r"((int)c) : "memory");
}
__device__ __forceinline__ void cp16_if(bool c, unsigned dst, const void *src) {
    asm volatile(EIK_PRED "2, 0; @p cp.async.cg.shared.global [%0], [%1], 16;}" ::"r"(dst), "l"(src), "r"((int)c)
                 : "memory");
}
__device__ __forceinline__ void cp16(unsigned dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// v = min(v, x) in the lanes where c holds
__device__ __forceinline__ void min_if(bool c, float &v, float x) {
    asm(EIK_PRED "2, 0; @p min.f32 %0, %0, %1;}" : "+f"(v) : "f"(x), "r"((int)c));
}
__device__ __forceinline__ void min_if(bool c, double &v, double x) {
    if (c) v = Num<double>::mn(v, x);
}
#undef EIK_PRED

// Shared control words of one engine run.
struct EngineCtl {
    long long lim;  // polls a wait may make (read once when the run starts)
    int *done;      // [nb] sweeps completed by the block (all rows written back)
    int *fin;       // [8] warps that finished sweep k (slot k & 7)
    int *chg;       // [8] any node changed in sweep k
    int *stop_at;   // first sweep that changed nothing (INT_MAX while unknown)
    int *abort_flag;
};

__device__ __forceinline__ int vload(const int *p) { return *(const volatile int *)p; }
__device__ __forceinline__ void vstore(int *p, int v) { *(volatile int *)p = v; }
template <bool GLOBAL>
__device__ __forceinline__ void fence() {
    if (GLOBAL) asm volatile("fence.acq_rel.gpu;" ::: "memory");
    else asm volatile("fence.acq_rel.cta;" ::: "memory");
}

// Bounded wait until ready() holds.  Returns false if the engine is stopping
// (the last useful sweep is known to precede `sweep`) or on timeout.
// Called by whole warps; the answer is the same in every lane.
template <class F>
__device__ __forceinline__ bool wait_until(F ready, const EngineCtl &C, int sweep, int *err) {
    if (__all_sync(FULL, ready())) return true;
    // the sleep doubles from 32 to 256 ns: short waits wake quickly, long ones
    // leave the issue slots to the warps doing work
    long long it = 0;
    unsigned ns = 32;
    while (!__all_sync(FULL, ready())) {
        if (__any_sync(FULL, vload(C.abort_flag) || vload(C.stop_at) < sweep)) return false;
        if (++it > C.lim) {
            vstore(C.abort_flag, 1);
            atomicExch(err, DEV_TIMEOUT);
            return false;
        }
        __nanosleep(ns);
        ns = ns < 256 ? 2 * ns : 256;
    }
    return true;
}

// FSM update u = min(u, u~) (Sec. 1.1, eq. FSMupdate) from the axis minima a, b.
// Static: r h, NaN at fixed nodes (Gamma) and outside the box, whose u~ is then
// NaN, so that they keep their value without a test.
template <class T>
struct FsmPolicy {
    static constexpr bool SYM = true;
    static __device__ __forceinline__ T pad() { return Num<T>::inf(); }
    static __device__ __forceinline__ T node(bool fixed, T r, T h) {
        return !fixed && r > T(0) ? Num<T>::mul(r, h) : Num<T>::nan();
    }
    __device__ __forceinline__ T update(T self, T a, T b, T rh, bool &changed) const {
        const T ut = local_solve2_min(a, b, rh);
        changed = Num<T>::below(ut, self);
        return changed ? ut : self;
    }
    // K independent nodes; their FP64 roots run together
    template <int K>
    __device__ __forceinline__ void update_all(const float *self, const float *a, const float *b, const float *rh,
                                               bool *changed, float *v) const {
#pragma unroll
        for (int j = 0; j < K; ++j) v[j] = update(self[j], a[j], b[j], rh[j], changed[j]);
    }
    template <int K>
    __device__ __forceinline__ void update_all(const double *self, const double *a, const double *b,
                                               const double *rh, bool *changed, double *v) const {
        Solve64 S[K];
        bool unsure = false;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            S[j] = solve2_start(a[j], b[j], rh[j]);
            unsure = unsure || S[j].root.unsure;
        }
        if (unsure) {
#pragma unroll
            for (int j = 0; j < K; ++j)
                if (S[j].root.unsure) root_decide(S[j].root, true);
        }
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const double ut = solve2_end(S[j]);
            changed[j] = Num<double>::below(ut, self[j]);
            v[j] = changed[j] ? ut : self[j];
        }
    }
};

// Shared memory of one warp (32-bit shared addresses).
struct WarpMem {
    unsigned ring, sring, halo, sbring;
};

// One sweep (number k, direction k mod 4) of physical block b by its warp.
// `hands`: the hand-off columns of all blocks ([nb][hand_elems(ny)], shared or,
// with GLOBAL, global memory).  Returns -1 if the engine is stopping, else
// whether any node changed.
//
// The work of a chunk boundary (write-back, copies, halo) is spread over the
// eight steps of the chunk, without branches, where it issues in the latency
// of the step's own chain; only the wait for the hand-in is between chunks.
template <bool GLOBAL, class T, int NST, bool HASB, class P>
__device__ int run_block(const Box<T, NST> &bx, const P &pol, int k, int b, const WarpMem &M, T *hands,
                         const EngineCtl &C, int *err) {
    constexpr int E = 16 / (int)sizeof(T);   // elements of a 16-byte access
    constexpr int VC = CH / E;               // 16-byte accesses per lane, chunk and static
    constexpr unsigned SZ = sizeof(T), ROWB = 32 * SZ, RMASK = RROWS * ROWB - 1;
    const T PAD = P::pad();
    const int dir = k & 3, sx = dir_sx(dir), sy = dir_sy(dir);
    const int lane = threadIdx.x & 31;
    const int NB = bx.nb, NY = bx.ny;
    const int q = sx > 0 ? b : NB - 1 - b;           // logical block
    const int pc = sx > 0 ? lane : 31 - lane;         // physical column in the block
    const int bp = b - sx, bn = b + sx;               // physical predecessor / successor
    const bool has_prev = bp >= 0 && bp < NB;
    const bool has_next = bn >= 0 && bn < NB;
    const bool lane0 = lane == 0, lane31 = lane == 31, low = lane < CH;
    const size_t he = hand_elems(NY);
    T *const hand_out = hands + (size_t)b * he;
    T *const hand_in = hands + (size_t)(has_prev ? bp : b) * he;
    const unsigned hand_out_s = GLOBAL ? 0u : (unsigned)__cvta_generic_to_shared(hand_out);
    const unsigned hand_in_s = GLOBAL ? 0u : (unsigned)__cvta_generic_to_shared(hand_in);
    const int nchunks = (NY + CH - 1) / CH;         // chunks of rows
    const int nJ = (NY + 31 + CH - 1) / CH;         // chunks of steps

    // Start condition: the successor block (whose old column this sweep reads)
    // has finished sweep k-1.  Our own block finished it in program order.
    if (k > 0 && has_next) {
        const int *dn = C.done + bn;
        if (!wait_until([&] { return vload(dn) >= k; }, C, k, err)) return -1;
        fence<GLOBAL>();
    }
    // When the x sign flipped, the column read as hand-in was read by the block
    // on the far side of the predecessor in sweep k-1: that block must have put
    // its NaNs back (it feeds the predecessor now, so this never waits longer
    // than the hand-in itself).  Otherwise this warp was the reader.
    if (k > 0 && !(k & 1) && bp - sx >= 0 && bp - sx < NB) {
        const int *dp = C.done + (bp - sx);
        if (!wait_until([&] { return vload(dp) >= k; }, C, k, err)) return -1;
        fence<GLOBAL>();
    }

    // u rows move between global memory and the ring in chunks of 8: this lane
    // copies 8 columns of row r8.  Chunks j and j + 8 share their ring rows.
    const int r8 = lane >> 2, cg = lane & 3;
    const int prow0 = sy > 0 ? 0 : NY - 1;            // physical row of logical row 0
    const int cstep = sy * CH * 32;                   // elements from one chunk to the next
    T *gcopy = bx.u + ((size_t)b * NY + prow0 + sy * r8) * 32 + cg * 8;  // chunk 0
    unsigned scopy = (unsigned)(prow0 + sy * r8) * ROWB + cg * 8 * SZ;
    int mcopy = r8;
    const int mfirst = k == 0 ? 0 : RROWS;            // first row not in the ring already
    auto issue_chunk = [&] {
        const unsigned dst = M.ring + (scopy & RMASK);
        const bool on = mcopy < NY && mcopy >= mfirst;
#pragma unroll
        for (int c = 0; c < 8 / E; ++c) cp16_if(on, dst + 16 * c, gcopy + c * E);
        gcopy += cstep;
        scopy += (unsigned)cstep * SZ;
        mcopy += CH;
    };
    uint4 wb[8 / E];
    auto wb_load = [&](unsigned off) {
#pragma unroll
        for (int c = 0; c < 8 / E; ++c)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(wb[c].x), "=r"(wb[c].y), "=r"(wb[c].z), "=r"(wb[c].w)
                         : "r"(M.ring + (off & RMASK) + 16 * c) : "memory");
    };
    auto wb_store = [&](int m, T *dst) {
#pragma unroll
        for (int c = 0; c < 8 / E; ++c) stcg16_if((unsigned)m < (unsigned)NY, dst + c * E, wb[c]);
    };
    // statics of 8 steps -> statics ring (slot = chunk mod SRCH)
    const size_t stbase = ((size_t)dir * NB + q) * bx.nstepp * 32;
    size_t stoff = stbase + lane * E;
    const uint8_t *sbp = HASB ? bx.sb + stbase + lane * 16 : nullptr;
    unsigned sslot = 0;
    auto issue_statics = [&] {
#pragma unroll
        for (int kk = 0; kk < NST; ++kk) {
            const unsigned dst = M.sring + (((unsigned)kk * SRCH + sslot) * CH * 32 + lane * E) * SZ;
#pragma unroll
            for (int c = 0; c < VC; ++c) cp16(dst + 512 * c, bx.st[kk] + stoff + c * 32 * E);
        }
        if (HASB) {
            cp16_if(lane < 16, M.sbring + sslot * CH * 32 + lane * 16, sbp);
            sbp += CH * 32;
        }
        stoff += CH * 32;
        sslot = sslot == SRCH - 1 ? 0 : sslot + 1;
    };
    // right neighbours of lane 31 in chunk j: logical rows 8j-31 .. 8j-24 of the
    // successor's first column, one row per lane, one chunk ahead in hreg
    const T *hsrc = bx.u + ((size_t)(has_next ? bn : b) * NY + prow0) * 32 + (sx > 0 ? 0 : 31) +
                    (ptrdiff_t)(sy * (lane - 31)) * 32;
    int mhalo = has_next && low ? lane - 31 : (1 << 29);
    T hreg = PAD;
    const unsigned shalo = M.halo + (lane & (CH - 1)) * SZ;
    auto load_halo = [&] {
        hreg = PAD;
        ldcg_if((unsigned)mhalo < (unsigned)NY, hsrc, hreg);
        hsrc += cstep;
        mhalo += CH;
    };

    // left neighbours of lane 0 in chunk j: rows 8j .. 8j+7 of the predecessor's
    // last column; with GLOBAL one row per lane (lanes 0..7), read a chunk ahead
    T hin[GLOBAL ? 1 : CH], hahead = PAD;
#pragma unroll
    for (int i = 0; i < (GLOBAL ? 1 : CH); ++i) hin[i] = PAD;
    const int hlim = has_prev ? NY : 0;  // rows there are to read
    auto hand_ahead = [&](int m0) { hand_ldg_if(low && m0 + lane < hlim, hand_in + m0 + lane, hahead); };
    auto hand_wait = [&](int m0) -> bool {
        if (GLOBAL) {
            hin[0] = hahead;
            hahead = PAD;
            bool again = false;
            return wait_until([&] {
                if (again) hand_ldg_if(low && m0 + lane < NY, hand_in + m0 + lane, hin[0]);
                again = true;
                return !(low && m0 + lane < NY && Hand<T>::is_empty(hin[0]));
            }, C, k, err);
        }
        const unsigned a = hand_in_s + m0 * SZ;
        return wait_until([&] {
#pragma unroll
            for (int c = 0; c < VC; ++c) hand_lds16(a + 16 * c, hin + (GLOBAL ? 0 : c * E));
            bool r = true;
#pragma unroll
            for (int i = 0; i < CH; ++i) r = r && (!Hand<T>::is_empty(hin[GLOBAL ? 0 : i]) || m0 + i >= NY);
            return r;
        }, C, k, err);
    };
    auto hand_clear = [&](int m0) {  // after every lane has read them
        if (GLOBAL) {
            hand_stg_if(low && m0 + lane < hlim, hand_in + m0 + lane, Hand<T>::empty());
        } else {
            hand_sts_if(low && m0 < hlim, hand_in_s + (m0 + (lane & (CH - 1))) * SZ, Hand<T>::empty());
        }
    };

    // Prologue: u chunks 0..LEAD-1 and statics chunks 0 and 1 in flight (one
    // group per chunk), halo of chunk 0 staged, of chunk 1 in hreg.
#pragma unroll
    for (int j = 0; j < LEAD; ++j) {
        issue_chunk();
        if (j < 2) issue_statics();
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    sts1_if(low, shalo, hreg);  // rows -31 .. -24
    hsrc += cstep;
    mhalo += CH;
    load_halo();
    if (has_prev) {
        if (GLOBAL) hand_ahead(0);
        if (!hand_wait(0)) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            return -1;
        }
        // the reader of our own column put its NaNs back in an earlier sweep,
        // before it wrote the value just read
        fence<GLOBAL>();
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();

    auto ok = [&](int m) { return (unsigned)m < (unsigned)NY; };
    // ring offsets (this lane's column) of its rows m, m+1, m+2 at step 0 (m = -lane)
    const unsigned rstep = (unsigned)(sy * (int)ROWB);
    unsigned roff = (unsigned)(prow0 - sy * lane) * ROWB + (unsigned)pc * SZ;
    unsigned a0 = M.ring + (roff & RMASK), a1 = M.ring + ((roff + rstep) & RMASK),
             a2 = M.ring + ((roff + 2 * rstep) & RMASK);
    roff = (roff + 2 * rstep) & RMASK;
    T cur = PAD, d1 = PAD, d2 = PAD;
    lds1_if(ok(-lane), a0, cur);
    lds1_if(ok(1 - lane), a1, d1);
    lds1_if(ok(2 - lane), a2, d2);
    T last = PAD, fromleft = PAD;                    // own previous result, the left lane's
    T fromright = __shfl_down_sync(FULL, d1, 1);     // the right lane's old value on this lane's row
    bool changed = false;
    // hand-out: lane 31's row at step s is s - 31
    const bool hands_out = has_next && lane31;
    unsigned ho_s = hand_out_s - 31 * SZ;
    T *ho_g = hand_out - 31;
    unsigned sread = 0;  // statics ring slot of this chunk

    for (int J = 0; J < nJ; ++J) {
        const int s0 = J * CH;
        T hal[CH];
#pragma unroll
        for (int c = 0; c < VC; ++c) lds16(M.halo + (J & 1) * CH * SZ + 16 * c, hal + c * E);
        uint2 sb8 = make_uint2(0u, 0u);
        if constexpr (HASB)
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(sb8.x), "=r"(sb8.y)
                         : "r"(M.sbring + sread * CH * 32 + lane * 8) : "memory");
        const unsigned sst = M.sring + (sread * CH * 32 + lane * E) * SZ;
        sread = sread == SRCH - 1 ? 0 : sread + 1;
        T sv[NST][E];  // statics of the current E steps
        // The chunk's 8 steps.  STEADY: every lane is on a valid row at every
        // step and so is the row three ahead that it loads, so the row tests
        // are dropped (the same operations on the same values otherwise).
        auto run_chunk = [&](auto steady_tag) {
            constexpr bool STEADY = decltype(steady_tag)::value;
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                const int m = s0 + i - lane;
                if (i % E == 0) {
#pragma unroll
                    for (int kk = 0; kk < NST; ++kk)
                        lds16(sst + (unsigned)kk * SRCH * CH * 32 * SZ + 512 * (i / E), sv[kk]);
                }
                // ---- boundary work of the chunk
                if (i == 0) {
                    wb_load(scopy);                                 // rows of chunk J-5
                    if (GLOBAL) hand_ahead(s0 + CH);
                }
                if (i == 1) wb_store(mcopy - RROWS, gcopy - 8 * (ptrdiff_t)cstep);
                if (i == 2) {
                    __syncwarp();
                    issue_chunk();       // u chunk J+LEAD, into the rows of chunk J-5
                    issue_statics();     // statics chunk J+2
                    asm volatile("cp.async.commit_group;" ::: "memory");
                }
                if (i == 3) {
                    hand_clear(s0);
                    sts1_if(low, shalo + ((J + 1) & 1) * CH * SZ, hreg);
                    load_halo();
                }
                // u chunk J+1 (first read at step 5) has landed
                if (i == 4) {
                    asm volatile("cp.async.wait_group 2;" ::: "memory");
                    __syncwarp();
                }
                // ---- the node
                T right = lane31 ? hal[i] : fromright;
                const T hl = GLOBAL ? __shfl_sync(FULL, hin[0], i) : hin[GLOBAL ? 0 : i];
                bool ch = false;
                T nw;
                if constexpr (P::SYM) {
                    min_if(lane0, right, hl);
                    min_if(!lane0, right, fromleft);
                    nw = pol.update(cur, right, Num<T>::mn(last, d1), sv[0][i % E], ch);
                } else {
                    const T left = lane0 ? hl : fromleft;
                    T s1[NST];
#pragma unroll
                    for (int kk = 0; kk < NST; ++kk) s1[kk] = sv[kk][i % E];
                    const uint8_t sbv = HASB ? (uint8_t)((i < 4 ? sb8.x : sb8.y) >> (8 * (i & 3))) : (uint8_t)0;
                    nw = pol.update(cur, sx > 0 ? left : right, sx > 0 ? right : left, sy > 0 ? last : d1,
                                    sy > 0 ? d1 : last, s1, sbv, ch);
                }
                if (!STEADY) nw = ok(m) ? nw : PAD;
                fromleft = __shfl_up_sync(FULL, nw, 1);
                if (STEADY) sts1(a0, nw);
                else sts1_if(ok(m), a0, nw);
                if (GLOBAL) hand_stg_if(hands_out && (STEADY || ok(m)), ho_g + i, nw);
                else hand_sts_if(hands_out && (STEADY || ok(m)), ho_s + i * SZ, nw);
                changed = changed || (ch && (STEADY || ok(m)));
                roff = (roff + rstep) & RMASK;
                const unsigned a3 = M.ring + roff;
                T d3 = PAD;
                if (STEADY) d3 = lds1(a3, T(0));
                else lds1_if(ok(m + 3), a3, d3);
                fromright = __shfl_down_sync(FULL, d2, 1);
                last = nw;
                cur = d1;
                d1 = d2;
                d2 = d3;
                a0 = a1;
                a1 = a2;
                a2 = a3;
            }
        };
        if (s0 >= 31 && s0 + CH + 2 < NY) run_chunk(std::true_type{});
        else run_chunk(std::false_type{});
        ho_s += CH * SZ;
        ho_g += CH;
        // statics of chunk J+1 have landed; every lane's rows and halo are visible
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        bool go = true;
        if (s0 + CH < hlim) go = hand_wait(s0 + CH);
        if (go && (J & 7) == 7) go = !__any_sync(FULL, vload(C.abort_flag) || vload(C.stop_at) < k);
        if (!go) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            return -1;
        }
    }
    // the last rows (gcopy, scopy and mcopy are at chunk nJ + LEAD; rows 64 back
    // share ring rows)
    for (int j = nJ >= 5 ? nJ - 5 : 0; j < nchunks; ++j) {
        const int back = nJ + LEAD - j;
        wb_load(scopy - (unsigned)(back * cstep) * SZ);
        wb_store(mcopy - back * CH, gcopy - (ptrdiff_t)back * cstep);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    fence<GLOBAL>();  // every lane's write-back before the block's completion flag
    __syncwarp();
    return __any_sync(FULL, changed) ? 1 : 0;
}

// What a run ended with, from its control words.  Final in the kernel itself only
// with one CTA: of several, the last to finish a sweep that was the last allowed may
// find that it changed nothing when the others have left already, so their result is
// read in a later kernel.
__device__ __forceinline__ void engine_result(const int *ctl, long long max_sweeps, long long &sweeps,
                                              bool &converged) {
    const int st = vload(ctl + 1);
    converged = st != 0x7fffffff && !vload(ctl);
    sweeps = st != 0x7fffffff ? (long long)st + 1 : max_sweeps;
}

// Runs sweeps on one box until a sweep changes nothing or max_sweeps ran.
// Single-CTA form (GLOBAL = false): the CTA holds every block of the box,
// blockDim.x >= 32 * bx.nb, engine_smem_bytes<T, NST, HASB>(nb, ny) bytes of
// dynamic shared memory at `smem`.  Multi-CTA form (GLOBAL = true): CTA c
// owns blocks [c * nw, c * nw + nw) with nw = blockDim.x / 32, hand-off
// columns live in `ghands` ([nb][hand_elems(ny)], every element Hand<T>::empty()
// before the launch) and the control words in `gctl` (engine_global_ints(nb)
// ints, set by engine_global_init before the launch); every CTA of the grid
// must be co-resident (cooperative launch).  All threads must call it.
template <class T, int NST, bool HASB, bool GLOBAL = false, class P>
__device__ void engine_run(const Box<T, NST> &bx, const P &pol, long long max_sweeps, char *smem, long long &sweeps,
                           bool &converged, int *err, T *ghands = nullptr, int *gctl = nullptr, int cta = -1) {
    const int nwc = GLOBAL ? (int)(blockDim.x >> 5) : bx.nb;   // warps (blocks) of this CTA
    // multi-CTA form: this CTA's index among the CTAs of the box (blockIdx.x
    // unless several boxes share the grid)
    const int b0 = GLOBAL ? (cta >= 0 ? cta : (int)blockIdx.x) * nwc : 0;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const size_t ring_b = (size_t)RROWS * 32 * sizeof(T);
    const size_t sring_b = (size_t)NST * SRCH * CH * 32 * sizeof(T);
    const size_t small_b = (size_t)2 * CH * sizeof(T);
    const size_t sb_b = HASB ? (size_t)SRCH * CH * 32 : 0;
    // layout: rings, statics rings, byte rings, halo, hand-off columns, control words; every part a multiple of 16 bytes
    char *const p_sring = smem + (size_t)nwc * ring_b;
    char *const p_sb = p_sring + (size_t)nwc * sring_b;
    char *const p_small = p_sb + (size_t)nwc * sb_b;
    char *const p_hand = p_small + (size_t)nwc * small_b;
    T *hands = GLOBAL ? ghands : reinterpret_cast<T *>(p_hand);
    const size_t he = hand_elems(bx.ny);
    int *ints = GLOBAL ? gctl : reinterpret_cast<int *>(p_hand + (size_t)nwc * he * sizeof(T));
    WarpMem M;
    M.ring = (unsigned)__cvta_generic_to_shared(smem + (size_t)warp * ring_b);
    M.sring = (unsigned)__cvta_generic_to_shared(p_sring + (size_t)warp * sring_b);
    M.sbring = (unsigned)__cvta_generic_to_shared(p_sb + (size_t)warp * sb_b);
    M.halo = (unsigned)__cvta_generic_to_shared(p_small + (size_t)warp * small_b);
    EngineCtl C;
    // polls here sleep 256 ns at most, a quarter of what the limit counts with
    const long long lim = spin_limit();
    C.lim = lim < (1ll << 60) ? 4 * lim : lim;
    C.abort_flag = ints;
    C.stop_at = ints + 1;
    C.fin = ints + 8;
    C.chg = ints + 16;
    C.done = ints + 32;

    if (!GLOBAL) {
        if (threadIdx.x == 0) {
            C.abort_flag[0] = 0;
            C.stop_at[0] = 0x7fffffff;
        }
        if (threadIdx.x < 8) {
            C.fin[threadIdx.x] = 0;
            C.chg[threadIdx.x] = 0;
        }
        if ((int)threadIdx.x < bx.nb) C.done[threadIdx.x] = 0;
        for (size_t i = threadIdx.x; i < (size_t)nwc * he; i += blockDim.x) hands[i] = Hand<T>::empty();
    }
    __syncthreads();

    const int b = b0 + warp;
    if (warp < nwc && b < bx.nb) {
        for (long long kk = 0; kk < max_sweeps; ++kk) {
            const int k = (int)kk;
            if (__any_sync(FULL, vload(C.abort_flag) || vload(C.stop_at) < k)) break;
            const int ch = run_block<GLOBAL, T, NST, HASB>(bx, pol, k, b, M, hands, C, err);
            if (ch < 0) break;
            // sweep k of this block is complete: publish it, then the sweep status
            if (lane == 0) {
                fence<GLOBAL>();
                vstore(C.done + b, k + 1);
                if (ch) atomicOr(C.chg + (k & 7), 1);
                fence<GLOBAL>();
                const int f = atomicAdd(C.fin + (k & 7), 1);
                if (f == bx.nb - 1) {
                    if (vload(C.chg + (k & 7)) == 0) {
                        atomicMin(C.stop_at, k);
                    } else {
                        vstore(C.chg + (k & 7), 0);
                        vstore(C.fin + (k & 7), 0);
                    }
                }
            }
            __syncwarp();
        }
    }
    __syncthreads();
    engine_result(ints, max_sweeps, sweeps, converged);
    __syncthreads();
}

// Sets the control words of a multi-CTA engine run (one thread block).
__device__ inline void engine_global_init(int *gctl, int nb) {
    for (int i = threadIdx.x; i < (int)engine_global_ints(nb); i += blockDim.x) gctl[i] = i == 1 ? 0x7fffffff : 0;
}

}  // namespace eik
