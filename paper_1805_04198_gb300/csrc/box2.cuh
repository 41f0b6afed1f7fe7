// box2.cuh -- Gauss-Seidel sweeps of a small 2-D box held in shared memory, by
// one warp.
//
// The same schedule as engine.cuh (any schedule that respects the four
// dependencies of a node gives the serial loop nest's result) without its
// chunks, copies and hand-offs: lane l owns the K columns K l .. K l + K - 1 (in
// the order of the sweep), column j of it is on row s - K l - j at step s, so
//  * the left neighbour (new) of column j is what column j - 1 produced one step
//    earlier, of column 0 what the left lane's last column did (a shuffle);
//  * the right neighbour (old) of column j is the value ahead of column j + 1, of
//    the last column the value ahead of the right lane's first (a shuffle);
//  * the neighbours along y are the column's own previous result and the value
//    ahead of it.
// A sweep takes NX + NY steps, whatever K is; the K local solves of a step are
// independent and hide each other's latency, and a second sweep starts at once.
// Rows outside the box are read as the guard rows -1 and NY, which like the
// padding columns stay +inf, their r h being NaN: u~ is never below the value and
// nothing is stored, so rows and columns need no tests.
//
// Shared memory: u and r h, [row -1 .. NY][P]; column K l + j stands at j * NL + l,
// so that neighbouring lanes, K rows and one column apart, are an odd number of
// words apart (K P is even) and a warp's accesses have no bank conflicts.
#pragma once

#include "engine.cuh"

namespace eik {

constexpr int BOX2_THREADS = 128;  // a CTA fills and empties the box; its first warp sweeps

// Columns per lane, lanes used and row pitch of a box nx columns wide.
__host__ __device__ inline int box2_k(int nx) { return (nx + 31) / 32; }
__host__ __device__ inline int box2_lanes(int nx) { return (nx + box2_k(nx) - 1) / box2_k(nx); }
__host__ __device__ inline int box2_pitch(int nx) {
    const int k = box2_k(nx), p = k * box2_lanes(nx);
    return (k & 1) ? (p + 1) & ~1 : p;
}
template <class T>
__host__ __device__ inline size_t box2_smem_bytes(int nx, int ny) {
    return (size_t)2 * (ny + 2) * box2_pitch(nx) * sizeof(T);
}

// Columns per lane with which a box is swept in this form, 0 = by the engine.
// Measured, us a sweep alone / 2432 boxes on the GPU, this form against the
// engine: FP32 17^2 2.7 / 5.1 against 5.8 / 9.4, 33^2 3.9 / 11.7 against 11.7 /
// 32.2, 65^2 8.8 / 32.6 against 16.3 / 66.7, 97^2 14.8 / 124 against 21.0 / 120,
// 129^2 (K = 5) 23 / 394 against 27 / 200.  FP64, where one warp has a quarter
// of an SM's FP64 rate (64 cycles an operation) and the engine's warps have all
// of it, whole grids: 17^2 266 us against 423, 32^2 520 / 675, 33^2 1078 / 1194,
// but 41^2 1386 / 1294, 64^2 3616 / 2644: up to 36 columns.  `most`: shared memory
// that leaves room for two boxes on an SM; a single box may take more.
template <class T>
__host__ __device__ constexpr int box2_kmax() { return sizeof(T) == 4 ? 4 : 2; }
template <class T>
__host__ __device__ inline int box2_use(int nx, int ny, size_t most = 100 << 10) {
    const int k = box2_k(nx);
    return k <= box2_kmax<T>() && (sizeof(T) == 4 || nx <= 36) && box2_smem_bytes<T>(nx, ny) <= most ? k : 0;
}

// Where the nodes of a box stand in its two shared arrays.
template <int K>
struct Box2 {
    int ny, nl, p;
    __device__ Box2(int nx, int ny_) : ny(ny_) {
        nl = (nx + K - 1) / K;
        p = (K & 1) ? (K * nl + 1) & ~1 : K * nl;
    }
    __device__ __forceinline__ int at(int x, int y) const {
        const int l = x / K;
        return (y + 1) * p + (x - l * K) * nl + l;
    }
    __device__ __forceinline__ int cells() const { return (ny + 2) * p; }
    // u +inf and r h NaN everywhere (all threads; a barrier must follow)
    template <class T>
    __device__ __forceinline__ void clear(T *su, T *sr) const {
        for (int i = threadIdx.x; i < cells(); i += blockDim.x) {
            su[i] = Num<T>::inf();
            sr[i] = Num<T>::nan();
        }
    }
};

// A boundary value in a box.  FP32 minima and comparisons pass over any NaN, and no
// hand-off column is at stake here, so it is stored as loaded: testing it makes the
// filling of the box wait for every load (64^2 subdomains 5.30 ms a solve, 5.17 so).
__device__ __forceinline__ float box2_gamma(float g) { return g; }
__device__ __forceinline__ double box2_gamma(double g) { return gamma_value(g); }

// Sweeps until one changes nothing or max_sweeps ran; called by one whole warp,
// the box filled and visible to it.  su and sr: shared addresses of u and r h.
template <int K, class T>
__device__ void box2_sweeps(const Box2<K> &B, unsigned su, unsigned sr, long long max_sweeps, long long &sweeps,
                            bool &conv) {
    using N = Num<T>;
    constexpr int SZ = (int)sizeof(T);
    const T INF = N::inf();
    const int lane = threadIdx.x & 31;
    const int NY = B.ny, NL = B.nl, P = B.p;
    const bool mine = lane < NL;
    const unsigned rel = sr - su;
    const int nsteps = NY + K * (NL - 1) + K - 1;
    FsmPolicy<T> pol;
    sweeps = 0;
    conv = false;
    for (long long kk = 0; kk < max_sweeps; ++kk) {
        const int dir = (int)(kk & 3), sx = dir_sx(dir), sy = dir_sy(dir);
        const int rstep = sy * P * SZ;
        // logical row 0 of the lane's columns (lanes without columns look at the
        // guard rows only, through column 0)
        unsigned base[K];
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const int l = mine ? (sx > 0 ? lane : NL - 1 - lane) : 0, jj = sx > 0 ? j : K - 1 - j;
            base[j] = su + (unsigned)(((sy > 0 ? 1 : NY) * P + jj * NL + l) * SZ);
        }
        T last[K], cur[K], nxt[K], rh[K];
        unsigned at[K];
        int m = mine ? -K * lane : (1 << 28);  // row of column 0; column j is on m - j
        auto addr = [&](int j, int row) -> unsigned {
            unsigned q = (unsigned)row;
            q = q < (unsigned)NY ? q : (unsigned)NY;  // rows before and after: the guard row NY
            return base[j] + q * (unsigned)rstep;
        };
#pragma unroll
        for (int j = 0; j < K; ++j) {
            last[j] = INF;
            at[j] = addr(j, m - j);
            cur[j] = lds1(at[j], T(0));
            rh[j] = lds1(at[j] + rel, T(0));
            nxt[j] = lds1(addr(j, m - j + 1), T(0));
        }
        T left = INF, right = __shfl_down_sync(FULL, nxt[0], 1);
        if (lane == 31) right = INF;
        bool changed = false;
#pragma unroll 4
        for (int s = 0; s < nsteps; ++s) {
            // loads for the next step
            unsigned a1[K];
            T n2[K], r1[K];
#pragma unroll
            for (int j = 0; j < K; ++j) {
                a1[j] = addr(j, m - j + 1);
                r1[j] = lds1(a1[j] + rel, T(0));
                n2[j] = lds1(addr(j, m - j + 2), T(0));
            }
            T v[K], a[K], b[K];
            bool ch[K];
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const T l = j > 0 ? last[j > 0 ? j - 1 : 0] : left;
                const T r = j + 1 < K ? nxt[j + 1 < K ? j + 1 : j] : right;
                a[j] = N::mn(l, r);
                b[j] = N::mn(last[j], nxt[j]);
            }
            pol.template update_all<K>(cur, a, b, rh, ch, v);
            left = __shfl_up_sync(FULL, v[K - 1], 1);
            right = __shfl_down_sync(FULL, n2[0], 1);
            if (lane == 0) left = INF;
            if (lane == 31) right = INF;
#pragma unroll
            for (int j = 0; j < K; ++j) {
                sts1_if(ch[j], at[j], v[j]);
                changed = changed || ch[j];
                last[j] = v[j];
                cur[j] = nxt[j];
                nxt[j] = n2[j];
                rh[j] = r1[j];
                at[j] = a1[j];
            }
            ++m;
        }
        ++sweeps;
        __syncwarp();
        if (!__any_sync(FULL, changed)) {
            conv = true;
            break;
        }
    }
}

}  // namespace eik
