// eik_fsm3.cu -- plain fast sweeping method on a whole 3-D grid (Sec. 1.1),
// the baseline the 3-D domain decomposition is compared against.
//
// Sweep k visits the nodes in ordering k mod 8 of the paper's loop nest (sign
// of x = bit 2, y = bit 1, z = bit 0); node (x, y, z) then reads the three
// neighbours before it already updated in this sweep and the others from
// before it.  Two schedules respect exactly those dependencies, with the update
// u = min(u, u~) by the 3-D Godunov local solve; the result is that of the
// serial loop nest.  Sweeps stop after the first one that changes nothing.
//
// k_fsm3_tiles: the columns along z are cut into 8 x 4 tiles, one warp per tile
// for the whole run, one column per lane, lane (i, j) on row s - i - j at step
// s: neighbours in x and y inside the tile by shuffles, z by walking.  Between
// tiles the new face columns are handed on through global memory, in columns
// whose unwritten elements hold a reserved NaN (the value is its own flag; the
// reader puts the NaN back); the old face of the next tile is read from its
// state, which it has finished in sweep k - 1.  All other data are the warp's
// own, loaded a chunk of steps ahead.  It is bound by the chain of a step along
// the wavefront (NX + NY + NZ steps and a hand-off per tile).
// 129 x 145 x 161 FP32: 92 ms in 55 sweeps with a grid barrier per hyperplane
// (3.9 us each), 9.5 ms so.
//
// k_fsm3_sweeps: hyperplanes of nodes with equal i + j + k, each updated by the
// whole GPU, a grid barrier between them; for grids with more tiles than warps
// fit on the GPU at once, and for workspaces without room for the tile form.  60 x 330 x 330 FP32: 254 ms (266 ms with the wind, which
// is not needed, worked out beside the value).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "host_util.h"
#include "prof.h"

namespace eik {

EIK_SPIN_LIMIT_SETTER(set_spin_limit_fsm3)

struct Fsm3Dev {
    unsigned long long sweeps;
    int converged;
    int err;
    unsigned bar[4];
    int chg[4];
};

template <class T>
struct Fsm3Args {
    const T *r;
    const uint8_t *gamma;
    const T *g;
    T *u;              // caller's output, strides sy, sz
    long long sy, sz;
    int nx, ny, nz;
    T h;
    T *w;              // state, [nz][ny][nx] or, in the tile form, [tile][z][32]
    T *rp;             // tile form: r h in the same order
    T *hand;           // tile form: hand-off columns, 4 x faces and 8 y faces per tile
    int *ctl;          // tile form: control words
    int ntx, nty, ntile;  // tiles in x and y; ntile = 0: hyperplane form
    Fsm3Dev *dev;
    long long max_sweeps;
    int launches;
};

template <class T>
__global__ void k_fsm3_init(Fsm3Args<T> A) {
    const size_t n = (size_t)A.nx * A.ny * A.nz;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(t % A.nx), y = (int)((t / A.nx) % A.ny), z = (int)(t / ((size_t)A.nx * A.ny));
        const size_t gi = (size_t)z * A.sz + (size_t)y * A.sy + x;
        A.w[t] = A.gamma[gi] ? gamma_value(A.g[gi]) : Num<T>::inf();  // Sec. 1.1 initialisation
    }
    if (blockIdx.x == 0 && threadIdx.x < 4) {
        A.dev->bar[threadIdx.x] = 0;
        A.dev->chg[threadIdx.x] = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.dev->err = 0;
        A.dev->sweeps = 0;
        A.dev->converged = 0;
    }
}

template <class T>
__global__ void k_fsm3_sweeps(Fsm3Args<T> A) {
    const long long wlim = spin_limit();  // limit of the grid-barrier waits
    const T INF = Num<T>::inf();
    const int nx = A.nx, ny = A.ny, nz = A.nz;
    const size_t plane = (size_t)nx * ny;
    const long long nthreads = (long long)gridDim.x * blockDim.x;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int ndiag = nx + ny + nz - 2;
    __shared__ int blk_ch;
    long long k = 0;
    bool conv = false;
    for (; k < A.max_sweeps; ++k) {
        const int q = (int)(k & 7);
        const int sx = (q & 4) ? 1 : -1, sy = (q & 2) ? 1 : -1, sz = (q & 1) ? 1 : -1;
        if (threadIdx.x == 0) blk_ch = 0;
        bool ch = false;
        for (int dg = 0; dg < ndiag; ++dg) {
            const int ilo = max(0, dg - (ny - 1) - (nz - 1)), ihi = min(nx - 1, dg);
            const long long ncand = (long long)(ihi - ilo + 1) * ny;
            for (long long c = tid; c < ncand; c += nthreads) {
                const int ip = ilo + (int)(c / ny), jp = (int)(c % ny), kp = dg - ip - jp;
                if (kp < 0 || kp >= nz) continue;
                const int x = sx > 0 ? ip : nx - 1 - ip;
                const int y = sy > 0 ? jp : ny - 1 - jp;
                const int z = sz > 0 ? kp : nz - 1 - kp;
                const size_t gi = (size_t)z * A.sz + (size_t)y * A.sy + x;
                if (A.gamma[gi]) continue;
                const size_t t = (size_t)z * plane + (size_t)y * nx + x;
                T vm[3], vp[3];
                vm[0] = x > 0 ? A.w[t - 1] : INF;
                vp[0] = x + 1 < nx ? A.w[t + 1] : INF;
                vm[1] = y > 0 ? A.w[t - nx] : INF;
                vp[1] = y + 1 < ny ? A.w[t + nx] : INF;
                vm[2] = z > 0 ? A.w[t - plane] : INF;
                vp[2] = z + 1 < nz ? A.w[t + plane] : INF;
                using N = Num<T>;
                const T ut = solve3(N::mn(vm[0], vp[0]), N::mn(vm[1], vp[1]), N::mn(vm[2], vp[2]), N::mul(A.r[gi], A.h));
                if (N::lowers(ut, A.w[t])) {
                    A.w[t] = ut;
                    ch = true;
                }
            }
            if (!grid_barrier(A.dev->bar, &A.dev->err, wlim)) return;
        }
        // sweep k changed something?  slot k % 3, cleared two sweeps ahead
        if (ch) blk_ch = 1;
        __syncthreads();
        if (threadIdx.x == 0 && blk_ch) atomicOr(&A.dev->chg[k % 3], 1);
        if (!grid_barrier(A.dev->bar, &A.dev->err, wlim)) return;
        const int any = *(volatile int *)&A.dev->chg[k % 3];
        if (blockIdx.x == 0 && threadIdx.x == 0) A.dev->chg[(k + 2) % 3] = 0;
        if (!any) {
            conv = true;
            ++k;
            break;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.dev->sweeps = (unsigned long long)(conv ? k : A.max_sweeps);
        A.dev->converged = conv ? 1 : 0;
    }
}

// --------------------------------------------------------------------------
// Tile form
// --------------------------------------------------------------------------
constexpr int T3CH = 4;       // steps per chunk
constexpr int T3WARPS = 4;    // warps (tiles) per CTA
constexpr int T3LAG = 10;     // steps by which the last lane of a tile is behind the first

// Elements of one hand-off column (index = row + i or row + j of the face lane).
__host__ __device__ inline int t3_col(int nz) { return (nz + T3LAG + T3CH) / T3CH * T3CH + T3CH; }

template <class T> struct T3NaN;
template <> struct T3NaN<float> {
    static __device__ __forceinline__ float empty() { return __uint_as_float(0x7fd5a5c3u); }
    static __device__ __forceinline__ bool is(float v) { return __float_as_uint(v) == 0x7fd5a5c3u; }
};
template <> struct T3NaN<double> {
    static __device__ __forceinline__ double empty() { return __longlong_as_double(0x7ffad5a5c3b4e1f7ll); }
    static __device__ __forceinline__ bool is(double v) { return bits64(v) == 0x7ffad5a5c3b4e1f7ll; }
};

// Predicated accesses (a branch around one costs more than the access).
#define EIK_P3 "{.reg .pred p; setp.ne.b32 p, %"
__device__ __forceinline__ void p3_ld(bool c, const float *a, float &v) {
    asm volatile(EIK_P3 "2, 0; @p ld.global.f32 %0, [%1];}" : "+f"(v) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_ld(bool c, const double *a, double &v) {
    asm volatile(EIK_P3 "2, 0; @p ld.global.f64 %0, [%1];}" : "+d"(v) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_ldnc(bool c, const float *a, float &v) {
    asm volatile(EIK_P3 "2, 0; @p ld.global.nc.f32 %0, [%1];}" : "+f"(v) : "l"(a), "r"((int)c));
}
__device__ __forceinline__ void p3_ldnc(bool c, const double *a, double &v) {
    asm volatile(EIK_P3 "2, 0; @p ld.global.nc.f64 %0, [%1];}" : "+d"(v) : "l"(a), "r"((int)c));
}
__device__ __forceinline__ void p3_ldcg(bool c, const float *a, float &v) {
    asm volatile(EIK_P3 "2, 0; @p ld.global.cg.f32 %0, [%1];}" : "+f"(v) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_ldcg(bool c, const double *a, double &v) {
    asm volatile(EIK_P3 "2, 0; @p ld.global.cg.f64 %0, [%1];}" : "+d"(v) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_st(bool c, float *a, float v) {
    asm volatile(EIK_P3 "2, 0; @p st.global.f32 [%0], %1;}" ::"l"(a), "f"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_st(bool c, double *a, double v) {
    asm volatile(EIK_P3 "2, 0; @p st.global.f64 [%0], %1;}" ::"l"(a), "d"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_sthand(bool c, float *a, float v) {
    asm volatile(EIK_P3 "2, 0; @p st.volatile.global.f32 [%0], %1;}" ::"l"(a), "f"(v), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_sthand(bool c, double *a, double v) {
    asm volatile(EIK_P3 "2, 0; @p st.volatile.global.f64 [%0], %1;}" ::"l"(a), "d"(v), "r"((int)c) : "memory");
}
// one chunk (T3CH elements, 16-byte aligned) of a hand-off column
__device__ __forceinline__ void p3_ldhand(bool c, const float *a, float *v) {
    asm volatile(EIK_P3 "5, 0; @p ld.volatile.global.v4.f32 {%0, %1, %2, %3}, [%4];}"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_ldhand(bool c, const double *a, double *v) {
    asm volatile(EIK_P3 "5, 0; @p ld.volatile.global.v2.f64 {%0, %1}, [%4]; @p ld.volatile.global.v2.f64 {%2, %3}, [%4+16];}"
                 : "+d"(v[0]), "+d"(v[1]), "+d"(v[2]), "+d"(v[3]) : "l"(a), "r"((int)c) : "memory");
}
__device__ __forceinline__ void p3_clhand(bool c, float *a, float e) {
    asm volatile(EIK_P3 "2, 0; @p st.volatile.global.v4.f32 [%0], {%1, %1, %1, %1};}" ::"l"(a), "f"(e), "r"((int)c)
                 : "memory");
}
__device__ __forceinline__ void p3_clhand(bool c, double *a, double e) {
    asm volatile(EIK_P3 "2, 0; @p st.volatile.global.v2.f64 [%0], {%1, %1}; @p st.volatile.global.v2.f64 [%0+16], {%1, %1};}"
                 ::"l"(a), "d"(e), "r"((int)c) : "memory");
}
#undef EIK_P3

template <class T>
__global__ void k_fsm3_pack(Fsm3Args<T> A) {
    // state and r h, [tile][z][32]: Sec. 1.1 initialisation; +inf and NaN outside the grid
    const size_t n = (size_t)A.ntile * A.nz * 32;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const int p = (int)(t & 31);
        const size_t row = t >> 5;
        const int b = (int)(row / A.nz), z = (int)(row - (size_t)b * A.nz);
        const int tx = b / A.nty, x = 8 * tx + (p & 7), y = 4 * (b - tx * A.nty) + (p >> 3);
        T v = Num<T>::inf(), rh = Num<T>::nan();
        if (x < A.nx && y < A.ny) {
            const size_t gi = (size_t)z * A.sz + (size_t)y * A.sy + x;
            const T r = A.r[gi];
            if (A.gamma[gi]) v = gamma_value(A.g[gi]);
            else if (r > T(0)) rh = Num<T>::mul(r, A.h);
        }
        A.w[t] = v;
        A.rp[t] = rh;
    }
    const size_t nh = (size_t)A.ntile * 12 * t3_col(A.nz);
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < nh; t += (size_t)gridDim.x * blockDim.x)
        A.hand[t] = T3NaN<T>::empty();
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < A.ntile + 32; t += gridDim.x * blockDim.x)
        A.ctl[t] = t == 1 ? 0x7fffffff : 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.dev->err = 0;
        A.dev->sweeps = 0;
        A.dev->converged = 0;
    }
}

// Control words: [0] abort, [1] first sweep that changed nothing, [8..15] tiles
// that finished sweep k (slot k & 7), [16..23] any change in sweep k, [32..]
// sweeps finished by each tile.
template <class T>
__device__ int fsm3_tile_sweep(const Fsm3Args<T> &A, int b, int k, long long wlim) {
    using N = Num<T>;
    const T INF = N::inf();
    const int q = k & 7;
    const int sx = (q & 4) ? 1 : -1, sy = (q & 2) ? 1 : -1, sz = (q & 1) ? 1 : -1;
    const int lane = threadIdx.x & 31, i = lane & 7, j = lane >> 3;
    const int nz = A.nz, ntx = A.ntx, nty = A.nty;
    const int tx = b / nty, ty = b - tx * nty;
    const int px = sx > 0 ? i : 7 - i, py = sy > 0 ? j : 3 - j;  // place in the tile
    const bool prevx = tx - sx >= 0 && tx - sx < ntx, nextx = tx + sx >= 0 && tx + sx < ntx;
    const bool prevy = ty - sy >= 0 && ty - sy < nty, nexty = ty + sy >= 0 && ty + sy < nty;
    volatile int *const ctl = A.ctl;
    volatile int *const done = A.ctl + 32;
    auto wait = [&](auto ready) -> bool {
        long long it = 0;
        unsigned ns = 32;
        while (!__all_sync(FULL, ready())) {
            if (__any_sync(FULL, ctl[0] != 0 || ctl[1] < k)) return false;
            if (++it > wlim) {
                ctl[0] = 1;
                atomicExch(&A.dev->err, DEV_TIMEOUT);
                return false;
            }
            __nanosleep(ns);
            ns = ns < 256 ? 2 * ns : 256;
        }
        return true;
    };
    if (k > 0) {
        // the tiles after this one, whose old faces are read, have finished sweep
        // k-1; and where the x (y) sign flipped, so has the tile on the far side of
        // the one before, which read that one's hand-off columns in sweep k-1 and
        // has put their NaNs back
        const bool fx = (q & 3) == 0 && tx - 2 * sx >= 0 && tx - 2 * sx < ntx;
        const bool fy = (q & 1) == 0 && ty - 2 * sy >= 0 && ty - 2 * sy < nty;
        if (!wait([&] {
                return (!nextx || done[b + sx * nty] >= k) && (!nexty || done[b + sy] >= k) &&
                       (!fx || done[b - 2 * sx * nty] >= k) && (!fy || done[b - 2 * sy] >= k);
            }))
            return -1;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
    }
    const int zs = sz * 32, z0 = sz > 0 ? 0 : nz - 1;
    const int own = py * 8 + px;
    const ptrdiff_t at0 = ((ptrdiff_t)b * nz + z0) * 32 + (ptrdiff_t)(-i - j) * zs;  // row of step 0
    T *wp = A.w + at0 + own;
    const T *rp = A.rp + at0 + own;
    // lanes 7 and rows 3 read the old face of the next tile, lanes 0 and rows 0
    // the hand-off columns of the one before
    const bool oldx = i == 7 && nextx, oldy = j == 3 && nexty, inx = i == 0 && prevx, iny = j == 0 && prevy;
    const T *oxp = A.w + at0 + (ptrdiff_t)(sx * nty) * nz * 32 + py * 8 + (sx > 0 ? 0 : 7);
    const T *oyp = A.w + at0 + (ptrdiff_t)sy * nz * 32 + (sy > 0 ? 0 : 24) + px;
    const size_t col = t3_col(nz);
    T *const hxs = A.hand, *const hys = A.hand + (size_t)A.ntile * 4 * col;
    T *hix = hxs + ((size_t)(prevx ? b - sx * nty : b) * 4 + py) * col;
    T *hiy = hys + ((size_t)(prevy ? b - sy : b) * 8 + px) * col;
    const bool outx = i == 7 && nextx, outy = j == 3 && nexty;
    T *hox = hxs + ((size_t)b * 4 + py) * col - 7;
    T *hoy = hys + ((size_t)b * 8 + px) * col - 3;
    auto ok = [&](int m) { return (unsigned)m < (unsigned)nz; };
    int m = -i - j;  // this lane's row at the first step of the chunk being loaded
    // data of the next chunk: the node ahead (old), r h, the x and y faces
    T nu[T3CH], nr[T3CH], nx[T3CH], ny[T3CH];
    auto load = [&] {
#pragma unroll
        for (int s = 0; s < T3CH; ++s) {
            nu[s] = nr[s] = nx[s] = ny[s] = INF;
            p3_ld(ok(m + s + 1), wp + (s + 1) * zs, nu[s]);
            p3_ldnc(ok(m + s), rp + s * zs, nr[s]);
            p3_ldcg(oldx && ok(m + s), oxp + s * zs, nx[s]);
            p3_ldcg(oldy && ok(m + s), oyp + s * zs, ny[s]);
        }
        p3_ldhand(inx, hix, nx);
        p3_ldhand(iny, hiy, ny);
    };
    auto ready = [&] {
        bool r = true;
#pragma unroll
        for (int s = 0; s < T3CH; ++s)
            r = r && !(ok(m + s) && ((inx && T3NaN<T>::is(nx[s])) || (iny && T3NaN<T>::is(ny[s]))));
        return r;
    };
    auto arrived = [&]() -> bool {
        bool again = false;
        return wait([&] {
            if (again) {
                p3_ldhand(inx, hix, nx);
                p3_ldhand(iny, hiy, ny);
            }
            again = true;
            return ready();
        });
    };
    const int nJ = (nz + T3LAG + T3CH - 1) / T3CH;
    T cur = INF, last = INF;
    p3_ld(ok(m), wp, cur);
    load();
    if (!arrived()) return -1;
    // the readers of this tile's columns put their NaNs back before they wrote the
    // values just read
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    bool changed = false;
    for (int J = 0; J < nJ; ++J) {
        T u[T3CH], r[T3CH], x[T3CH], y[T3CH];
#pragma unroll
        for (int s = 0; s < T3CH; ++s) {
            u[s] = nu[s];
            r[s] = nr[s];
            x[s] = nx[s];
            y[s] = ny[s];
        }
        T *const w0 = wp, *const ox0 = hox, *const oy0 = hoy;
        const int m0 = m;
        __syncwarp();
        p3_clhand(inx, hix, T3NaN<T>::empty());
        p3_clhand(iny, hiy, T3NaN<T>::empty());
        wp += T3CH * zs;
        rp += T3CH * zs;
        oxp += T3CH * zs;
        oyp += T3CH * zs;
        hix += T3CH;
        hiy += T3CH;
        hox += T3CH;
        hoy += T3CH;
        m += T3CH;
        if (J + 1 < nJ) load();
#pragma unroll
        for (int s = 0; s < T3CH; ++s) {
            const T nxt = u[s];
            T xm = __shfl_up_sync(FULL, last, 1), ym = __shfl_up_sync(FULL, last, 8);
            T xp = __shfl_down_sync(FULL, nxt, 1), yp = __shfl_down_sync(FULL, nxt, 8);
            if (i == 0) xm = x[s];
            if (i == 7) xp = x[s];
            if (j == 0) ym = y[s];
            if (j == 3) yp = y[s];
            const bool on = ok(m0 + s);
            const T ut = solve3(N::mn(xm, xp), N::mn(ym, yp), N::mn(last, nxt), r[s]);
            const bool ch = on && N::lowers(ut, cur);
            const T v = ch ? ut : cur;
            p3_sthand(outx && on, ox0 + s, v);
            p3_sthand(outy && on, oy0 + s, v);
            p3_st(ch, w0 + s * zs, v);
            changed = changed || ch;
            last = on ? v : INF;
            cur = nxt;
        }
        bool go = true;
        if (J + 1 < nJ) go = arrived();
        if (go && (J & 15) == 15) go = !__any_sync(FULL, ctl[0] != 0 || ctl[1] < k);
        if (!go) return -1;
    }
    asm volatile("fence.acq_rel.gpu;" ::: "memory");  // every lane's values before the tile's completion
    __syncwarp();
    return __any_sync(FULL, changed) ? 1 : 0;
}

template <class T>
__global__ void __launch_bounds__(32 * T3WARPS, sizeof(T) == 4 ? 4 : 3) k_fsm3_tiles(Fsm3Args<T> A) {
    const long long wlim = spin_limit();
    const int b = blockIdx.x * T3WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= A.ntile) return;
    volatile int *const ctl = A.ctl;
    for (long long kk = 0; kk < A.max_sweeps; ++kk) {
        const int k = (int)kk;
        if (__any_sync(FULL, ctl[0] != 0 || ctl[1] < k)) break;
        const int ch = fsm3_tile_sweep(A, b, k, wlim);
        if (ch < 0) break;
        if (lane == 0) {
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            ctl[32 + b] = k + 1;
            if (ch) atomicOr(&A.ctl[16 + (k & 7)], 1);
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            if (atomicAdd(&A.ctl[8 + (k & 7)], 1) == A.ntile - 1) {
                if (ctl[16 + (k & 7)] == 0) {
                    atomicMin(&A.ctl[1], k);
                } else {
                    ctl[16 + (k & 7)] = 0;
                    ctl[8 + (k & 7)] = 0;
                }
            }
        }
        __syncwarp();
    }
}

template <class T>
__global__ void k_fsm3_out(Fsm3Args<T> A, eik_fsm_stats *out) {
    const size_t n = (size_t)A.nx * A.ny * A.nz;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const size_t row = t / A.nx;
        const int x = (int)(t - row * A.nx), z = (int)(row / A.ny), y = (int)(row - (size_t)z * A.ny);
        size_t src = t;
        if (A.ntile) src = ((size_t)((x >> 3) * A.nty + (y >> 2)) * A.nz + z) * 32 + (y & 3) * 8 + (x & 7);
        A.u[(size_t)z * A.sz + (size_t)y * A.sy + x] = A.w[src];
    }
    if (out && blockIdx.x == 0 && threadIdx.x == 0) {
        unsigned long long sweeps = A.dev->sweeps;
        int conv = A.dev->converged;
        if (A.ntile) {
            const int st = A.ctl[1];
            conv = st != 0x7fffffff && !A.ctl[0];
            sweeps = st != 0x7fffffff ? (unsigned long long)st + 1 : (unsigned long long)A.max_sweeps;
        }
        out->sweeps = (int64_t)sweeps;
        out->converged = conv;
        out->error = A.dev->err;
        out->updates = (int64_t)sweeps * A.nx * A.ny * A.nz;
        out->launches = A.launches;
    }
}

// Tiles that can be co-resident on the 152 SMs (5 CTAs of k_fsm3_tiles on an SM in
// FP32, 3 in FP64): larger grids are swept by hyperplanes, whatever the workspace.
template <class T>
constexpr size_t T3MOST = (size_t)152 * T3WARPS * (sizeof(T) == 4 ? 5 : 3);

static size_t fsm3_tile_count(const eik_grid *grid) {
    return (size_t)((grid->n[0] + 7) / 8) * ((grid->n[1] + 3) / 4);
}

// The workspace of the tile form or of the hyperplane form, which needs the state
// only (257^3 FP64: 136 MB; with tiles 2.5 times as much).
template <class T>
static size_t fsm3_layout(const eik_grid *grid, bool tiles, Fsm3Args<T> *A, void *ws) {
    const size_t ntx = (grid->n[0] + 7) / 8, nty = (grid->n[1] + 3) / 4, nt = ntx * nty;
    const size_t cells = nt * 32 * grid->n[2];
    Carver cv(ws);
    if (!tiles) {
        T *w = cv.take<T>((size_t)grid->n[0] * grid->n[1] * grid->n[2]);
        Fsm3Dev *dev = cv.take<Fsm3Dev>(1);
        if (A) {
            A->w = w;
            A->dev = dev;
        }
        return cv.used + 256;
    }
    T *w = cv.take<T>(cells), *rp = cv.take<T>(cells);
    T *hand = cv.take<T>(nt * 12 * t3_col((int)grid->n[2]));
    int *ctl = cv.take<int>(nt + 32);
    Fsm3Dev *dev = cv.take<Fsm3Dev>(1);
    if (A) {
        A->w = w;
        A->rp = rp;
        A->hand = hand;
        A->ctl = ctl;
        A->dev = dev;
        A->ntx = (int)ntx;
        A->nty = (int)nty;
    }
    return cv.used + 256;
}

template <class T>
static size_t fsm3_size(const eik_grid *grid, bool least) {
    return fsm3_layout<T>(grid, !least && fsm3_tile_count(grid) <= T3MOST<T>, nullptr, nullptr);
}

// least = false: the workspace to ask for; true: what a solve can do with
size_t fsm3_workspace_size(const eik_grid *grid, bool least) {
    return grid->dtype == EIK_F64 ? fsm3_size<double>(grid, least) : fsm3_size<float>(grid, least);
}

template <class T>
static int fsm3_run_t(const eik_grid *grid, const void *r, const uint8_t *gamma, const void *g, void *u,
                      int64_t max_sweeps, void *ws, size_t ws_bytes, eik_fsm_stats *stats, cudaStream_t s) {
    Fsm3Args<T> A;
    memset(&A, 0, sizeof(A));
    A.r = static_cast<const T *>(r);
    A.gamma = gamma;
    A.g = static_cast<const T *>(g);
    A.u = static_cast<T *>(u);
    A.sy = grid->stride[1];
    A.sz = grid->stride[2];
    A.nx = (int)grid->n[0];
    A.ny = (int)grid->n[1];
    A.nz = (int)grid->n[2];
    A.h = (T)grid->h;
    A.max_sweeps = max_sweeps;
    A.launches = 3;
    int rc, dev, nsm = 0;
    if ((rc = cuda_check(cudaGetDevice(&dev), "cudaGetDevice"))) return rc;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const size_t n = (size_t)A.nx * A.ny * A.nz;
    const int eb = (int)std::min<size_t>((n + 255) / 256, (size_t)nsm * 16);
    int per_sm = 0, tok;
    void *args[] = {&A};
    if ((rc = cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fsm3_tiles<T>, 32 * T3WARPS, 0),
                         "occupancy")))
        return rc;
    const size_t tiles = fsm3_tile_count(grid), ctas = (tiles + T3WARPS - 1) / T3WARPS;
    const bool tile_form = tiles <= T3MOST<T> && ctas <= (size_t)per_sm * nsm &&
                           ws_bytes >= fsm3_layout<T>(grid, true, nullptr, nullptr);
    fsm3_layout<T>(grid, tile_form, &A, ws);
    if (tile_form) {
        A.ntile = (int)tiles;
        EIK_LAUNCH("fsm3_init", s, k_fsm3_pack<T><<<eb, 256, 0, s>>>(A));
        tok = prof_begin("fsm3_sweeps", s);
        rc = cuda_check(cudaLaunchCooperativeKernel((void *)k_fsm3_tiles<T>, (int)ctas, 32 * T3WARPS, args, 0, s),
                        "fsm3 cooperative launch");
    } else {
        const int threads = 512;
        if ((rc = cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fsm3_sweeps<T>, threads, 0),
                             "occupancy")))
            return rc;
        // one or two CTAs per SM keep the grid barrier short
        const int blocks = std::max(1, std::min(per_sm, 2) * nsm);
        EIK_LAUNCH("fsm3_init", s, k_fsm3_init<T><<<eb, 256, 0, s>>>(A));
        tok = prof_begin("fsm3_sweeps", s);
        rc = cuda_check(cudaLaunchCooperativeKernel((void *)k_fsm3_sweeps<T>, blocks, threads, args, 0, s),
                        "fsm3 cooperative launch");
    }
    prof_end(tok, s);
    if (rc) return rc;
    EIK_LAUNCH("fsm3_out", s, k_fsm3_out<T><<<eb, 256, 0, s>>>(A, stats));
    return cuda_check(cudaGetLastError(), "fsm3 launch");
}

int fsm3_run(const eik_grid *grid, const void *r, const uint8_t *gamma, const void *g, void *u, int64_t max_sweeps,
             void *ws, size_t ws_bytes, eik_fsm_stats *stats, cudaStream_t s) {
    if (grid->dtype == EIK_F64) return fsm3_run_t<double>(grid, r, gamma, g, u, max_sweeps, ws, ws_bytes, stats, s);
    return fsm3_run_t<float>(grid, r, gamma, g, u, max_sweeps, ws, ws_bytes, stats, s);
}

}  // namespace eik
