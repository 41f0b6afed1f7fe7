// eik_dd3.cu -- the two-scale DD iteration (Sec. 3.2, Steps 1-4, Alg. 1-5)
// in three dimensions.  The paper states the method in 2-D and says it
// "can be generalized"; the generalisation used here:
//   * coarse set: every node with some index = 0 mod c, the union of the
//     c^3 - (c-1)^3 shifted coarse grids (offsets with at least one zero);
//   * Alg. 4 / Alg. 5 agreement tests on every interface / coarse-line axis
//     of a node; the causal sweep (Alg. 2) along every axis e whose fine
//     neighbours stay on the coarse set (the node lies on a coarse plane of
//     another axis);
//   * the 3-D Godunov local solve (sorted-minima cascade).
// Subdomains and shifted coarse grids are small boxes that fit in shared
// memory, so each is swept by one CTA along hyperplanes i + j + k = const
// (nodes of a hyperplane are independent; a barrier separates hyperplanes),
// which is the serial Gauss-Seidel order of the paper's loop nest.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "host_util.h"
#include "prof.h"

namespace eik {

EIK_SPIN_LIMIT_SETTER(set_spin_limit_dd3)

struct Grid3 {
    int ox, oy, oz, mx, my, mz;
    long long off;  // element offset in the coarse arrays ([z][y][x] box)
};

struct DD3Geom {
    int n[3], T[3], S[3], c, ng;
    long long nc;           // coarse elements
    double h, H;
};

struct DevStats3 {
    unsigned long long fsm_sweeps_max, coarse_sweeps_max, fsm_caps, coarse_caps, fine_updates, coarse_updates;
    unsigned long long fine_skips;
    int causal_rounds_max, err, iters, converged;
};

template <class T>
struct DD3Args {
    DD3Geom G;
    const T *r;
    const uint8_t *gamma;
    const T *g;
    T *u_out;
    long long sy, sz;
    T *rp;            // r h of the subdomains, [subdomain][column tile][z][32]; null without room for it
    int fpx, fps, fo, gpx, gps, go;  // layout (see Box3) of the subdomain and the shifted-grid boxes
    Grid3 *grids;
    int *offmap;  // [c^3] offset -> grid index (-1 if not a shifted grid)
    T *U, *Uprev, *U0, *rc, *uk, *cold;
    uint8_t *W, *wk, *mask;
    T *cu;
    uint8_t *cw;
    int *done;
    double *deltas;
    int *chg;
    uint8_t *lflag;  // causal sweep: lines to walk again; null without room: all of them
    unsigned *bar;
    DevStats3 *st;
    // Step 2 data of each subdomain's last solve in this call (the starting
    // value of every face node and the coarse wind an inflow node echoes),
    // [ntiles][face slots], and whether the subdomain has been solved
    T *sig_u;
    uint8_t *sig_w;
    int *sig_ok;
    T theta, tol;
    // constant weight 0: Alg. 5 yields u^k at every node, Alg. 4 writes
    // U^{k+1} = u^k itself and Step 4 is not launched
    int step4_identity;
    int max_iter;
    long long max_fsm, max_coarse;
    // per-node weight of Sec. 4.2 (adaptive = 1): weights, damping, cap, the
    // last four C_H(nbrs U) (slot m % 4), du = u^k - u^{k-1}, the weight
    int adaptive;
    double om[3], sg, sd, sx0, cap;
    T *Ch[4];
    double *du;
    T *th;
};

template <class T>
__device__ __forceinline__ size_t fidx(const DD3Args<T> &A, int X, int Y, int Z) {
    return (size_t)Z * A.sz + (size_t)Y * A.sy + X;
}

template <class T>
__device__ __forceinline__ long long coarse_addr3(const DD3Args<T> &A, int X, int Y, int Z) {
    const int c = A.G.c;
    const int g = A.offmap[((Z % c) * c + (Y % c)) * c + (X % c)];
    const Grid3 d = A.grids[g];
    return d.off + ((long long)(Z / c) * d.my + (Y / c)) * d.mx + (X / c);
}

__device__ __forceinline__ int coarse_axes3(int X, int Y, int Z, int c) {
    return (X % c == 0 ? 1 : 0) | (Y % c == 0 ? 2 : 0) | (Z % c == 0 ? 4 : 0);
}

// --------------------------------------------------------------------------
// Box sweeps in shared memory along hyperplanes.  Sweep k uses ordering
// k mod 8 of the paper's loop nest: sign of x = bit 2, y = bit 1, z = bit 0.
// Hyperplane i + j + k = dg (logical indices of the ordering) holds one node of
// each (x, y) column, and its nodes are independent of each other.
//
// The columns are cut into 8 x 4 tiles, one column per lane, and a warp takes
// two tiles next to each other in y, whose local solves are independent and
// interleave: they have nodes on mz + 14 hyperplanes and the warp passes over
// the others.  A lane
// walks its column, so the node behind is its previous result and the node
// ahead becomes its next one; the four other neighbours come from shared
// memory, whose row and plane pitches (box3_pitch) put a tile's 32 nodes of a
// hyperplane into different banks.  The read-only data of a node are loaded
// two hyperplanes ahead.
//
// A barrier separates hyperplanes (flags between neighbouring warps instead of
// the barrier: 25% more instructions, 161 ms against 129 ms).  The kernel
// is bound by the issue of the local solves (about 95 instructions a node) and,
// on the first and last hyperplanes of a sweep, by the latency of a few warps.
// Subdomain stage of the 257^3 solve (512 boxes of 33^3, 27 iterations): 120 ms
// (three tiles on 16 warps 129 ms); 267 ms with 32 columns of a row per warp,
// stepped through on every hyperplane.
//
// The policy gives a cursor along a column, load_if(on, cursor, places ahead,
// Stat) and apply(self, minus sides, plus sides, Stat, changed).
// --------------------------------------------------------------------------
constexpr int BOX3_SLOTS = 2;      // tiles per warp with prefetched data
constexpr int BOX3_THREADS = 768;  // threads of a box-sweep CTA

// The shared memory by which a box (mx x my x mz) is accepted or refused: the
// documented size limit.  The bordered layout may take more, up to what
// box3_pitch is given, the layout without border takes less.
__host__ inline size_t box3_limit(int mx, int my, int mz, size_t tsz) {
    return (size_t)mz * (mx * my + ((mx * my) & 1)) * (tsz + 1) + 16;
}

// Layout of a box in shared memory: node (x, y, z) at z * ps + (y + 1) * px + x + 1
// with px > mx and ps >= (my + 1) * px, so that every row and every plane is
// followed by cells that stay +inf and missing x and y neighbours need no test.
// px and ps are the smallest with the fewest bank conflicts within a tile.  A
// thin box whose border does not fit is stored without (px = mx), its columns
// at the sides then test for their neighbours.
__host__ __device__ inline size_t box3_elems(int mx, int mz, int px, int ps) {
    return (size_t)mz * ps + (px > mx ? px + 2 : 0);
}
__host__ inline void box3_pitch(int mx, int my, int mz, int tsz, size_t bytes, int &px, int &ps) {
    int best = 1 << 30;
    px = mx + 1;
    ps = (my + 1) * px;
    for (int x = mx + 1; x <= mx + 8; ++x)
        for (int add = 0; add < 32; ++add) {
            const int p = x * (my + 1) + add;
            if (box3_elems(mx, mz, x, p) * tsz + 16 > bytes) break;
            // lanes served together: 32 words, or 16 of 8 bytes
            const int group = 128 / tsz;
            int worst = 0;
            for (int g0 = 0; g0 < 32; g0 += group) {
                int cnt[32] = {0};
                for (int l = g0; l < g0 + group; ++l) {
                    const int i = l & 7, j = l >> 3;
                    const int w = ((i + j * x - (i + j) * p) % group + group) % group;
                    worst = std::max(worst, ++cnt[w]);
                }
            }
            if (worst < best || (worst == best && p < ps)) {
                best = worst;
                px = x;
                ps = p;
            }
        }
    if (best == 1 << 30) {
        px = mx;
        ps = mx * my;
    }
}

// `o` = offset of node (0, 0, 0): px + 1, or 0 without border
template <class T>
struct Box3 {
    T *su;
    int mx, my, mz, px, ps, o;
    __device__ __forceinline__ int at(int x, int y, int z) const { return z * ps + y * px + x + o; }
    __device__ __forceinline__ void node(int e, int &x, int &y, int &z) const {
        const int row = e / mx;
        x = e - row * mx;
        z = row / my;
        y = row - z * my;
    }
    // neighbours of node (x, y, z), +inf where missing
    __device__ __forceinline__ void nbrs(int x, int y, int z, T *vm, T *vp) const {
        const T INF = Num<T>::inf();
        const int q = at(x, y, z);
        const bool b = o != 0;
        vm[0] = b || x > 0 ? su[q - 1] : INF;
        vp[0] = b || x + 1 < mx ? su[q + 1] : INF;
        vm[1] = b || y > 0 ? su[q - px] : INF;
        vp[1] = b || y + 1 < my ? su[q + px] : INF;
        vm[2] = z > 0 ? su[q - ps] : INF;
        vp[2] = z + 1 < mz ? su[q + ps] : INF;
    }
    // every cell +inf (all threads; a barrier must follow)
    __device__ __forceinline__ void clear() const {
        const int n = mz * ps + (o ? px + 2 : 0);
        for (int i = threadIdx.x; i < n; i += blockDim.x) su[i] = Num<T>::inf();
    }
};

// Four shared-memory values of the lanes where c holds (others keep theirs).
__device__ __forceinline__ void lds4_if(bool c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, float *v) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %8, 0; @p ld.shared.f32 %0, [%4]; @p ld.shared.f32 %1, [%5]; "
                 "@p ld.shared.f32 %2, [%6]; @p ld.shared.f32 %3, [%7];}"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"((int)c)
                 : "memory");
}
__device__ __forceinline__ void lds4_if(bool c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, double *v) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %8, 0; @p ld.shared.f64 %0, [%4]; @p ld.shared.f64 %1, [%5]; "
                 "@p ld.shared.f64 %2, [%6]; @p ld.shared.f64 %3, [%7];}"
                 : "+d"(v[0]), "+d"(v[1]), "+d"(v[2]), "+d"(v[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"((int)c)
                 : "memory");
}
__device__ __forceinline__ void lds_if(bool c, unsigned a, float &v) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %2, 0; @p ld.shared.f32 %0, [%1];}" : "+f"(v) : "r"(a), "r"((int)c)
                 : "memory");
}
__device__ __forceinline__ void lds_if(bool c, unsigned a, double &v) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %2, 0; @p ld.shared.f64 %0, [%1];}" : "+d"(v) : "r"(a), "r"((int)c)
                 : "memory");
}
__device__ __forceinline__ void ldg_if(bool c, const float *a, float &v) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %2, 0; @p ld.global.nc.f32 %0, [%1];}" : "+f"(v) : "l"(a), "r"((int)c));
}
__device__ __forceinline__ void ldg_if(bool c, const double *a, double &v) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %2, 0; @p ld.global.nc.f64 %0, [%1];}" : "+d"(v) : "l"(a), "r"((int)c));
}
__device__ __forceinline__ void sts_if(bool c, unsigned a, float v) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %2, 0; @p st.shared.f32 [%0], %1;}" ::"r"(a), "f"(v), "r"((int)c)
                 : "memory");
}
__device__ __forceinline__ void sts_if(bool c, unsigned a, double v) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %2, 0; @p st.shared.f64 [%0], %1;}" ::"r"(a), "d"(v), "r"((int)c)
                 : "memory");
}

__host__ __device__ inline int box3_tiles(int mx, int my) { return ((mx + 7) >> 3) * ((my + 3) >> 2); }

template <class T, class P>
__device__ void box3_sweeps(const Box3<T> &B, const P &pol, long long max_sweeps, long long &sweeps, bool &conv) {
    using S = typename P::Stat;
    const T INF = Num<T>::inf();
    T *const su = B.su;
    const int mx = B.mx, my = B.my, mz = B.mz, ps = B.ps, px = B.px;
    const int ndiag = mx + my + mz - 2;
    const int nty = (my + 3) >> 2, nt = box3_tiles(mx, my);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    auto column = [&](int tile, int &x, int &y) {  // tiles in y order
        const int tx = tile / nty, ty = tile - tx * nty;
        x = 8 * tx + (lane & 7);
        y = 4 * ty + (lane >> 3);
        return tile < nt && x < mx && y < my;
    };
    int cx[BOX3_SLOTS], cy[BOX3_SLOTS];
    bool cv[BOX3_SLOTS];
#pragma unroll
    for (int t = 0; t < BOX3_SLOTS; ++t) cv[t] = column(warp * BOX3_SLOTS + t, cx[t], cy[t]);
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(su);
    constexpr int SZ = (int)sizeof(T);
    sweeps = 0;
    conv = false;
    for (long long k = 0; k < max_sweeps; ++k) {
        const int q = (int)(k & 7);
        const int sx = (q & 4) ? 1 : -1, sy = (q & 2) ? 1 : -1, sz = (q & 1) ? 1 : -1;
        const int zstep = sz * ps * SZ, z0 = sz > 0 ? 0 : mz - 1;
        int kp[BOX3_SLOTS];              // position of the column's node along z, on the current hyperplane
        int lo = 1 << 28, hi = 0;        // hyperplanes of the warp's tiles
        unsigned at[BOX3_SLOTS];         // shared address of that node
        T cur[BOX3_SLOTS], last[BOX3_SLOTS], nb[BOX3_SLOTS][4];
        S sa[BOX3_SLOTS], sb[BOX3_SLOTS];      // data of the even and the odd hyperplanes
        typename P::Cursor pc[BOX3_SLOTS];
#pragma unroll
        for (int t = 0; t < BOX3_SLOTS; ++t) {
            // logical x + y of the column
            const int base = cv[t] ? (sx > 0 ? cx[t] : mx - 1 - cx[t]) + (sy > 0 ? cy[t] : my - 1 - cy[t]) : (1 << 28);
            lo = min(lo, base);
            hi = max(hi, cv[t] ? base + mz : 0);
            kp[t] = -base;
            at[t] = sbase + (unsigned)(cv[t] ? B.at(cx[t], cy[t], z0) * SZ - base * zstep : 0);
            cur[t] = last[t] = INF;
#pragma unroll
            for (int i = 0; i < 4; ++i) nb[t][i] = INF;
            sa[t] = sb[t] = P::none();
            // (a lane without a column has no place to count from)
            pc[t] = pol.cursor(cv[t] ? cx[t] : 0, cv[t] ? cy[t] : 0, warp * BOX3_SLOTS + t, lane, z0, sz,
                               cv[t] ? -base : 0);
            pol.load_if((unsigned)kp[t] < (unsigned)mz, pc[t], 0, sa[t]);
            pol.load_if((unsigned)(kp[t] + 1) < (unsigned)mz, pc[t], 1, sb[t]);
            if (base == 0) cur[t] = su[B.at(cx[t], cy[t], z0)];  // a lane on its first node at hyperplane 0
        }
        lo = __reduce_min_sync(FULL, lo);
        hi = __reduce_max_sync(FULL, hi);
        bool ch = false;
        auto plane = [&](int dg, S *st) {
            if (dg + 2 >= lo && dg < hi) {  // uniform in the warp
                // gather, solve, store (nodes of one hyperplane never read each other)
                bool in[BOX3_SLOTS], c1[BOX3_SLOTS];
                T nxt[BOX3_SLOTS], v[BOX3_SLOTS];
#pragma unroll
                for (int t = 0; t < BOX3_SLOTS; ++t) {
                    in[t] = (unsigned)kp[t] < (unsigned)mz;
                    const unsigned a = at[t];
                    if (B.o) {
                        lds4_if(in[t], a - SZ, a + SZ, a - px * SZ, a + px * SZ, nb[t]);
                    } else {  // (a missing neighbour's value stays +inf)
                        lds_if(in[t] && cx[t] > 0, a - SZ, nb[t][0]);
                        lds_if(in[t] && cx[t] + 1 < mx, a + SZ, nb[t][1]);
                        lds_if(in[t] && cy[t] > 0, a - px * SZ, nb[t][2]);
                        lds_if(in[t] && cy[t] + 1 < my, a + px * SZ, nb[t][3]);
                    }
                    nxt[t] = INF;
                    lds_if((unsigned)(kp[t] + 1) < (unsigned)mz, a + zstep, nxt[t]);
                }
#pragma unroll
                for (int t = 0; t < BOX3_SLOTS; ++t) {
                    const T va[3] = {nb[t][0], nb[t][2], sz > 0 ? last[t] : nxt[t]};
                    const T vb[3] = {nb[t][1], nb[t][3], sz > 0 ? nxt[t] : last[t]};
                    c1[t] = false;
                    v[t] = pol.apply(cur[t], va, vb, st[t], c1[t]);
                    c1[t] = c1[t] && in[t];
                }
#pragma unroll
                for (int t = 0; t < BOX3_SLOTS; ++t) {
                    sts_if(c1[t], at[t], v[t]);
                    ch = ch || c1[t];
                    last[t] = in[t] ? v[t] : INF;
                    cur[t] = nxt[t];
                    pol.load_if((unsigned)(kp[t] + 2) < (unsigned)mz, pc[t], 2, st[t]);
                }
            }
#pragma unroll
            for (int t = 0; t < BOX3_SLOTS; ++t) {
                ++kp[t];
                at[t] += (unsigned)zstep;
                pol.advance(pc[t]);
            }
            // tiles beyond the prefetched ones (wide boxes)
            for (int tile = BOX3_SLOTS * nw + warp; tile < nt; tile += nw) {
                int x, y;
                if (!column(tile, x, y)) continue;
                const int k1 = dg - ((sx > 0 ? x : mx - 1 - x) + (sy > 0 ? y : my - 1 - y));
                if ((unsigned)k1 < (unsigned)mz) {
                    const int z = z0 + sz * k1;
                    T va[3], vb[3];
                    B.nbrs(x, y, z, va, vb);
                    S s1 = P::none();
                    pol.load_if(true, pol.cursor(x, y, tile, lane, z, sz, 0), 0, s1);
                    bool c1 = false;
                    const T v = pol.apply(su[B.at(x, y, z)], va, vb, s1, c1);
                    if (c1) su[B.at(x, y, z)] = v;
                    ch = ch || c1;
                }
            }
            __syncthreads();
        };
        for (int dg = 0; dg < ndiag; dg += 2) {
            plane(dg, sa);
            if (dg + 1 < ndiag) plane(dg + 1, sb);
        }
        ++sweeps;
        if (!__syncthreads_or(ch ? 1 : 0)) {
            conv = true;
            break;
        }
    }
}

// FSM update (Sec. 1.1): u = min(u, u~), from r h (NaN at fixed nodes, whose u~
// is then never below their value).
template <class T>
struct Fsm3Update {
    using Stat = T;
    static __device__ __forceinline__ T none() { return Num<T>::nan(); }
    __device__ __forceinline__ T apply(T self, const T *vm, const T *vp, T rh, bool &changed) const {
        using N = Num<T>;
        const T ut = solve3(N::mn(vm[0], vp[0]), N::mn(vm[1], vp[1]), N::mn(vm[2], vp[2]), rh);
        changed = N::lowers(ut, self);
        return changed ? ut : self;
    }
};
// r h of a subdomain, packed [column tile][z][32] (k3_pack_tiles)
template <class T>
struct Fsm3Tile : Fsm3Update<T> {
    const T *rp;
    int mz;
    // element of the column's node `kp0` places before its first one in z order
    struct Cursor {
        int at, step;
    };
    __device__ __forceinline__ Cursor cursor(int, int, int tile, int lane, int z0, int sz, int kp0) const {
        return Cursor{((tile * mz + z0) * 32 + lane) + kp0 * sz * 32, sz * 32};
    }
    __device__ __forceinline__ void advance(Cursor &c) const { c.at += c.step; }
    __device__ __forceinline__ void load_if(bool on, const Cursor &c, int ahead, T &v) const {
        ldg_if(on, rp + c.at + ahead * c.step, v);
    }
};
// The same from the caller's arrays, for a workspace without room for the packed
// copy (73^3 FP64, 3^3 subdomains of 25^3: 89 ms a solve, packed 74 ms).
template <class T>
struct Fsm3Direct : Fsm3Update<T> {
    const T *r;  // at the subdomain's first node
    const uint8_t *gamma;
    long long sy, sz;
    T h;
    struct Cursor {
        long long at, step;
    };
    __device__ __forceinline__ Cursor cursor(int x, int y, int, int, int z0, int dz, int kp0) const {
        return Cursor{x + y * sy + (z0 + (long long)kp0 * dz) * sz, dz * sz};
    }
    __device__ __forceinline__ void advance(Cursor &c) const { c.at += c.step; }
    __device__ __forceinline__ void load_if(bool on, const Cursor &c, int ahead, T &v) const {
        if (on) {
            const long long f = c.at + ahead * c.step;
            v = !gamma[f] && r[f] > T(0) ? Num<T>::mul(r[f], h) : Num<T>::nan();
        }
    }
};
// r of a shifted grid in box order (<= 0 at fixed nodes)
template <class T>
struct Fsm3Grid : Fsm3Update<T> {
    const T *rc;
    int mx, my;
    T Hs;
    struct Cursor {
        int at, step;
    };
    __device__ __forceinline__ Cursor cursor(int x, int y, int, int, int z0, int sz, int kp0) const {
        const int plane = mx * my;
        return Cursor{z0 * plane + y * mx + x + kp0 * sz * plane, sz * plane};
    }
    __device__ __forceinline__ void advance(Cursor &c) const { c.at += c.step; }
    __device__ __forceinline__ void load_if(bool on, const Cursor &c, int ahead, T &v) const {
        if (on) {
            const T r = rc[c.at + ahead * c.step];
            v = r > T(0) ? Num<T>::mul(r, Hs) : Num<T>::nan();
        }
    }
};

// Alg. 5 update on a shifted grid box (box layout arrays from `off`).
template <class T>
struct Alg5_3 {
    const T *rc, *uk, *cold;
    const uint8_t *mask;
    long long off;
    int mx, my;
    T Hs, theta;
    const T *th;  // per-node weight (nullptr: the constant theta)
    struct Stat {
        T rc, uk, cold, th;
        uint8_t m;
    };
    static __device__ __forceinline__ Stat none() { return Stat{T(1), T(0), T(0), T(0), 1}; }
    struct Cursor {
        int at, step;
    };
    __device__ __forceinline__ Cursor cursor(int x, int y, int, int, int z0, int sz, int kp0) const {
        const int plane = mx * my;
        return Cursor{z0 * plane + y * mx + x + kp0 * sz * plane, sz * plane};
    }
    __device__ __forceinline__ void advance(Cursor &c) const { c.at += c.step; }
    __device__ __forceinline__ void load_if(bool on, const Cursor &c, int ahead, Stat &v) const {
        if (on) {
            const long long a = off + c.at + ahead * c.step;
            v = Stat{rc[a], uk[a], cold[a], th ? th[a] : theta, mask[a]};
        }
    }
    __device__ __forceinline__ T apply(T self, const T *vm, const T *vp, const Stat &st, bool &changed) const {
        using N = Num<T>;
        const uint8_t m = st.m;
        changed = false;
        if (m & 1) return self;
        uint8_t w;
        const T Ut = local_solve3(vm, vp, N::mul(st.rc, Hs), w);
        const T ukv = st.uk, cv = st.cold;
        bool pass = (Ut < N::inf()) && (cv < N::inf());
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            const int wc = wind_comp(w, ax);
            pass = pass && ((wc <= 0 && (m & (2 << (2 * ax)))) || (wc >= 0 && (m & (4 << (2 * ax)))));
        }
        const T nu = pass ? N::add(ukv, N::mul(st.th, N::sub(Ut, cv))) : ukv;
        changed = !(nu == self);
        return nu;
    }
};

// --------------------------------------------------------------------------
// Set-up
// --------------------------------------------------------------------------
template <class T>
__global__ void k3_init(DD3Args<T> A) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        memset(A.st, 0, sizeof(DevStats3));
        *A.done = 0;
        A.bar[0] = A.bar[1] = 0;
    }
    for (int k = threadIdx.x; k < A.max_iter + 2; k += blockDim.x) A.deltas[k] = k == 0 ? INFINITY : 0.0;
    for (int t = threadIdx.x; t < A.G.T[0] * A.G.T[1] * A.G.T[2]; t += blockDim.x) A.sig_ok[t] = 0;
}

// one CTA row per shifted grid (blockIdx.y), threads over its nodes
template <class T>
__global__ void k3_pack_coarse(DD3Args<T> A) {
    const Grid3 d = A.grids[blockIdx.y];
    const long long n = (long long)d.mx * d.my * d.mz;
    const int c = A.G.c;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e % d.mx), j = (int)((e / d.mx) % d.my), k = (int)(e / ((long long)d.mx * d.my));
        const int X = d.ox + c * i, Y = d.oy + c * j, Z = d.oz + c * k;
        const size_t f = fidx(A, X, Y, Z);
        const bool gam = A.gamma[f] != 0;
        const long long a = d.off + e;
        A.rc[a] = gam ? T(-1) : A.r[f];
        A.U0[a] = gam ? gamma_value(A.g[f]) : Num<T>::inf();
        A.W[a] = WIND_ZERO;
    }
}

// r h of every subdomain in column-tile order (NaN at Gamma and outside).
template <class T>
__global__ void k3_pack_tiles(DD3Args<T> A) {
    const DD3Geom &G = A.G;
    const int mx = G.S[0] + 1, my = G.S[1] + 1, mz = G.S[2] + 1;
    const int nty = (my + 3) >> 2, nt = box3_tiles(mx, my);
    const int tile = blockIdx.x;
    const int t0 = tile % G.T[0], t1 = (tile / G.T[0]) % G.T[1], t2 = tile / (G.T[0] * G.T[1]);
    const int n = nt * mz * 32;
    const T hs = T(G.h);
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int lane = e & 31, row = e >> 5, ct = row / mz, z = row - ct * mz;
        const int tx = ct / nty, x = 8 * tx + (lane & 7), y = 4 * (ct - tx * nty) + (lane >> 3);
        T v = Num<T>::nan();
        if (x < mx && y < my) {
            const size_t f = fidx(A, t0 * G.S[0] + x, t1 * G.S[1] + y, t2 * G.S[2] + z);
            const T r = A.r[f];
            if (!A.gamma[f] && r > T(0)) v = Num<T>::mul(r, hs);
        }
        A.rp[(size_t)tile * n + e] = v;
    }
}

template <class T>
__device__ void grid3_winds(const DD3Args<T> &A, const Grid3 &d, const Box3<T> &B, T Hs) {
    const T INF = Num<T>::inf();
    const int n = d.mx * d.my * d.mz;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        int x, y, z;
        B.node(e, x, y, z);
        const long long a = d.off + e;
        uint8_t w = WIND_ZERO;
        const T rv = A.rc[a];
        if (rv > T(0) && B.su[B.at(x, y, z)] < INF) {
            T vm[3], vp[3];
            B.nbrs(x, y, z, vm, vp);
            (void)local_solve3(vm, vp, Num<T>::mul(rv, Hs), w);
        }
        A.W[a] = w;
    }
}

// Step 1: FSM with Alg. 1 on every shifted grid (one CTA per grid).
template <class T>
__global__ void __launch_bounds__(BOX3_THREADS, 1) k3_step1(DD3Args<T> A) {
    extern __shared__ __align__(16) char smem[];
    const Grid3 d = A.grids[blockIdx.x];
    const int n = d.mx * d.my * d.mz;
    const Box3<T> B{reinterpret_cast<T *>(smem), d.mx, d.my, d.mz, A.gpx, A.gps, A.go};
    T *const su = B.su;
    auto sq = [&](int e) {
        int x, y, z;
        B.node(e, x, y, z);
        return B.at(x, y, z);
    };
    B.clear();
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += blockDim.x) su[sq(e)] = A.U0[d.off + e];
    __syncthreads();
    Fsm3Grid<T> pol;
    pol.rc = A.rc + d.off;
    pol.mx = d.mx;
    pol.my = d.my;
    pol.Hs = T(A.G.H);
    long long sweeps;
    bool conv;
    box3_sweeps(B, pol, A.max_coarse, sweeps, conv);
    for (int e = threadIdx.x; e < n; e += blockDim.x) A.U[d.off + e] = su[sq(e)];
    grid3_winds(A, d, B, T(A.G.H));
    if (threadIdx.x == 0) {
        atomicMax(&A.st->coarse_sweeps_max, (unsigned long long)sweeps);
        if (!conv) atomicAdd(&A.st->coarse_caps, 1ull);
        atomicAdd(&A.st->coarse_updates, (unsigned long long)sweeps * n);
    }
}

// Step 4: Alg. 5 on every shifted grid.
template <class T>
__global__ void __launch_bounds__(BOX3_THREADS, 1) k3_step4(DD3Args<T> A, int k) {
    if (*A.done) return;
    extern __shared__ __align__(16) char smem[];
    const Grid3 d = A.grids[blockIdx.x];
    const int n = d.mx * d.my * d.mz;
    const T Hs = T(A.G.H);
    const Box3<T> B{reinterpret_cast<T *>(smem), d.mx, d.my, d.mz, A.gpx, A.gps, A.go};
    T *const su = B.su;
    auto sq = [&](int e) {
        int x, y, z;
        B.node(e, x, y, z);
        return B.at(x, y, z);
    };
    B.clear();
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += blockDim.x) su[sq(e)] = A.U[d.off + e];
    __syncthreads();
    // C_H(nbrs^H(U^k)) and U^k for the delta
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        int x, y, z;
        B.node(e, x, y, z);
        const long long a = d.off + e;
        A.Uprev[a] = su[B.at(x, y, z)];
        T vm[3], vp[3];
        B.nbrs(x, y, z, vm, vp);
        const T rv = A.rc[a];
        uint8_t w;
        const T cold = local_solve3(vm, vp, Num<T>::mul(rv > T(0) ? rv : T(0), Hs), w);
        A.cold[a] = cold;
        if (A.adaptive) {
            // Sec. 4.2 with every term lagged as in eq. firstthetaest
            double thv = (double)A.theta;
            if (k >= 1) {
                const int nt = k < 3 ? k : 3;
                const T *c1 = A.Ch[(k + 3) & 3], *c2 = A.Ch[(k + 2) & 3], *c3 = A.Ch[(k + 1) & 3];
                double dC[3] = {0.0, 0.0, 0.0};
                dC[0] = __dsub_rn((double)cold, (double)c1[a]);
                if (nt > 1) dC[1] = __dsub_rn((double)c1[a], (double)c2[a]);
                if (nt > 2) dC[2] = __dsub_rn((double)c2[a], (double)c3[a]);
                thv = theta_estimate(A, A.du[a], dC, nt, (double)A.theta);
            }
            A.Ch[k & 3][a] = cold;
            A.th[a] = (T)thv;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += blockDim.x) su[sq(e)] = A.U0[d.off + e];  // Sec. 1.1 initialisation
    __threadfence_block();
    __syncthreads();
    Alg5_3<T> pol{A.rc, A.uk, A.cold, A.mask, d.off, d.mx, d.my, Hs, A.theta, A.adaptive ? A.th : nullptr};
    long long sweeps;
    bool conv;
    box3_sweeps(B, pol, A.max_coarse, sweeps, conv);
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        A.U[d.off + e] = su[sq(e)];
        A.W[d.off + e] = A.wk[d.off + e];  // W = w^k
    }
    if (threadIdx.x == 0) {
        atomicMax(&A.st->coarse_sweeps_max, (unsigned long long)sweeps);
        if (!conv) atomicAdd(&A.st->coarse_caps, 1ull);
        atomicAdd(&A.st->coarse_updates, (unsigned long long)sweeps * n);
    }
}

// --------------------------------------------------------------------------
// Steps 2 + 3: one CTA per subdomain, the subdomain box in shared memory.
// --------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ bool tile3_inflow(const DD3Args<T> &A, const int *l, const int *Xg, long long &ca) {
    bool face = false;
    for (int a = 0; a < 3; ++a) face = face || l[a] == 0 || l[a] == A.G.S[a];
    if (!face) return false;
    ca = coarse_addr3(A, Xg[0], Xg[1], Xg[2]);
    const uint8_t w = A.W[ca];
    bool in = false;
    for (int a = 0; a < 3; ++a) {
        const int wc = wind_comp(w, a);
        in = in || (l[a] == 0 && wc > 0) || (l[a] == A.G.S[a] && wc < 0);
    }
    return in;
}

// Face slots of a subdomain box: the six face planes in the order x = 0,
// x = S, y = 0, y = S, z = 0, z = S; a node on several faces takes the slot
// of the first.  Returns -1 off the faces.
__host__ __device__ inline int box3_face_slots(const int *S) {
    const int m0 = S[0] + 1, m1 = S[1] + 1, m2 = S[2] + 1;
    return 2 * (m1 * m2 + m0 * m2 + m0 * m1);
}
__device__ inline int box3_face_slot(const int *S, const int *l) {
    const int m0 = S[0] + 1, m1 = S[1] + 1, m2 = S[2] + 1;
    if (l[0] == 0) return l[1] + m1 * l[2];
    if (l[0] == S[0]) return m1 * m2 + l[1] + m1 * l[2];
    int off = 2 * m1 * m2;
    if (l[1] == 0) return off + l[0] + m0 * l[2];
    if (l[1] == S[1]) return off + m0 * m2 + l[0] + m0 * l[2];
    off += 2 * m0 * m2;
    if (l[2] == 0) return off + l[0] + m0 * l[1];
    if (l[2] == S[2]) return off + m0 * m1 + l[0] + m0 * l[1];
    return -1;
}

template <class T>
__device__ __forceinline__ bool same_bits3(T a, T b);
template <>
__device__ __forceinline__ bool same_bits3<float>(float a, float b) { return __float_as_uint(a) == __float_as_uint(b); }
template <>
__device__ __forceinline__ bool same_bits3<double>(double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b);
}

template <class T, bool PACKED>
__global__ void __launch_bounds__(BOX3_THREADS, 1) k3_fine(DD3Args<T> A) {
    if (*A.done) return;
    extern __shared__ __align__(16) char smem[];
    const DD3Geom &G = A.G;
    const int tile = blockIdx.x;
    const int t0 = tile % G.T[0], t1 = (tile / G.T[0]) % G.T[1], t2 = tile / (G.T[0] * G.T[1]);
    const int mx = G.S[0] + 1, my = G.S[1] + 1, mz = G.S[2] + 1;
    const int n = mx * my * mz;
    const T INF = Num<T>::inf();
    const Box3<T> B{reinterpret_cast<T *>(smem), mx, my, mz, A.fpx, A.fps, A.fo};
    T *const su = B.su;
    const int b0 = t0 * G.S[0], b1 = t1 * G.S[1], b2 = t2 * G.S[2];
    // Step 2: boundary data; inflow nodes start at U (and are swept like the
    // rest), interior and outflow nodes at +inf; Gamma is fixed at g.  The
    // face nodes' data are compared with those of the subdomain's previous
    // solve in this call: if none changed, that solve's results (fine values,
    // copies) are still in place and equal bit for bit to what this one would
    // write (r, Gamma and g do not change within a call), so it is skipped.
    const int nslot = box3_face_slots(G.S);
    T *sgu = A.sig_u + (size_t)tile * nslot;
    uint8_t *sgw = A.sig_w + (size_t)tile * nslot;
    bool diff = false;
    B.clear();
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        int l[3];
        B.node(e, l[0], l[1], l[2]);
        const int Xg[3] = {b0 + l[0], b1 + l[1], b2 + l[2]};
        const size_t f = fidx(A, Xg[0], Xg[1], Xg[2]);
        long long ca;
        T v = INF;
        uint8_t fixed = 0;
        if (A.gamma[f]) {
            v = gamma_value(A.g[f]);
            fixed = 1;
        } else if (tile3_inflow(A, l, Xg, ca)) {
            v = A.U[ca];
            fixed = 2;
        }
        su[B.at(l[0], l[1], l[2])] = v;
        const int fs = box3_face_slot(G.S, l);
        if (fs >= 0) {
            const T sv = fixed ? v : INF;
            const uint8_t swv = fixed == 2 ? A.W[ca] : (uint8_t)0;
            if (!same_bits3(sv, sgu[fs]) || swv != sgw[fs]) {
                diff = true;
                sgu[fs] = sv;
                sgw[fs] = swv;
            }
        }
    }
    const bool solved = A.sig_ok[tile] != 0;
    if (!__syncthreads_or(diff) && solved) {
        if (threadIdx.x == 0) atomicAdd(&A.st->fine_skips, 1ull);
        return;
    }
    if (threadIdx.x == 0) A.sig_ok[tile] = 1;
    __syncthreads();
    long long sweeps;
    bool conv;
    if constexpr (PACKED) {
        Fsm3Tile<T> pol;
        pol.rp = A.rp + (size_t)tile * box3_tiles(mx, my) * mz * 32;
        pol.mz = mz;
        box3_sweeps(B, pol, A.max_fsm, sweeps, conv);
    } else {
        Fsm3Direct<T> pol;
        const size_t f = fidx(A, b0, b1, b2);
        pol.r = A.r + f;
        pol.gamma = A.gamma + f;
        pol.sy = A.sy;
        pol.sz = A.sz;
        pol.h = T(G.h);
        box3_sweeps(B, pol, A.max_fsm, sweeps, conv);
    }
    if (threadIdx.x == 0) {
        atomicMax(&A.st->fsm_sweeps_max, (unsigned long long)sweeps);
        if (!conv) atomicAdd(&A.st->fsm_caps, 1ull);
        atomicAdd(&A.st->fine_updates, (unsigned long long)sweeps * n);
    }
    // outputs: copies (u, w) at coarse-set nodes, fine values elsewhere
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        int l[3];
        B.node(e, l[0], l[1], l[2]);
        const int Xg[3] = {b0 + l[0], b1 + l[1], b2 + l[2]};
        const size_t f = fidx(A, Xg[0], Xg[1], Xg[2]);
        const T uv = su[B.at(l[0], l[1], l[2])];
        if (!coarse_axes3(Xg[0], Xg[1], Xg[2], G.c)) {
            A.u_out[f] = uv;
            continue;
        }
        const long long ca = coarse_addr3(A, Xg[0], Xg[1], Xg[2]);
        uint8_t w = WIND_ZERO;
        const bool fixed = A.gamma[f] != 0;
        long long ca2;
        if (!fixed && tile3_inflow(A, l, Xg, ca2) && uv == A.U[ca]) {
            w = A.W[ca] | WIND_ECHO;  // inflow value kept: the coarse wind
        } else if (!fixed && uv < INF) {
            T vm[3], vp[3];
            B.nbrs(l[0], l[1], l[2], vm, vp);
            (void)local_solve3(vm, vp, Num<T>::mul(A.r[f], T(G.h)), w);
        }
        int slot = 0;
        for (int a = 0; a < 3; ++a)
            if (Xg[a] % G.S[a] == 0 && Xg[a] > 0 && Xg[a] < G.n[a] - 1 && l[a] == 0) slot |= 1 << a;
        A.cu[(size_t)slot * G.nc + ca] = uv;
        A.cw[(size_t)slot * G.nc + ca] = w;
    }
}

// --------------------------------------------------------------------------
// Alg. 4 and the inputs of Alg. 5
// --------------------------------------------------------------------------
template <class T>
__global__ void k3_alg4(DD3Args<T> A) {
    if (*A.done) return;
    const DD3Geom &G = A.G;
    const Grid3 d = A.grids[blockIdx.y];
    const long long n = (long long)d.mx * d.my * d.mz;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int Xg[3] = {d.ox + G.c * (int)(e % d.mx), d.oy + G.c * (int)((e / d.mx) % d.my),
                           d.oz + G.c * (int)(e / ((long long)d.mx * d.my))};
        const long long a = d.off + e;
        int B = 0;
        for (int ax = 0; ax < 3; ++ax)
            if (Xg[ax] % G.S[ax] == 0 && Xg[ax] > 0 && Xg[ax] < G.n[ax] - 1) B |= 1 << ax;
        const uint8_t Wk = A.W[a];
        int best = 0;
        if (B) {
            int sel = 0;
            bool ok = true;
            for (int ax = 0; ax < 3 && ok; ++ax) {
                if (!(B & (1 << ax))) continue;
                bool allneg = wind_comp(Wk, ax) <= 0, allpos = wind_comp(Wk, ax) >= 0;
                for (int s = 0; s < 8; ++s) {
                    if (s & ~B) continue;
                    const int wv = wind_comp(A.cw[(size_t)s * G.nc + a], ax);
                    if (wv > 0) allneg = false;
                    if (wv < 0) allpos = false;
                }
                // Alg. 4: wind toward -axis -> plus-side copy (first branch)
                if (allneg) sel |= 1 << ax;
                else if (!allpos) ok = false;
            }
            if (ok) {
                best = sel;
            } else {
                // minimum of the fine solutions: copies that echo their Step 2
                // value are candidates only if every copy does; ties keep the
                // lowest subdomain index (slot order)
                bool computed = false;
                for (int s = 0; s < 8; ++s)
                    if (!(s & ~B) && !(A.cw[(size_t)s * G.nc + a] & WIND_ECHO)) computed = true;
                best = -1;
                T bv = T(0);
                for (int s = 0; s < 8; ++s) {
                    if (s & ~B) continue;
                    if (computed && (A.cw[(size_t)s * G.nc + a] & WIND_ECHO)) continue;
                    const T v = A.cu[(size_t)s * G.nc + a];
                    if (best < 0 || v < bv) {
                        bv = v;
                        best = s;
                    }
                }
            }
        }
        const T ukv = A.cu[(size_t)best * G.nc + a];
        const uint8_t wkv = A.cw[(size_t)best * G.nc + a] & (uint8_t)~WIND_ECHO;
        if (A.adaptive) A.du[a] = __dsub_rn((double)ukv, (double)A.uk[a]);  // u^k - u^{k-1}
        A.uk[a] = ukv;
        A.wk[a] = wkv;
        const size_t f = fidx(A, Xg[0], Xg[1], Xg[2]);
        A.u_out[f] = ukv;
        if (A.step4_identity) {
            // Step 4 with weight 0: U^{k+1} = u^k before the causal sweep, W = w^k
            A.Uprev[a] = A.U[a];
            A.U[a] = ukv;
            A.W[a] = wkv;
            continue;
        }
        uint8_t m = A.gamma[f] ? 1 : 0;
        for (int ax = 0; ax < 3; ++ax) {
            const bool on = Xg[ax] % G.c == 0;
            const int wf = wind_comp(wkv, ax), wc = wind_comp(Wk, ax);
            if (!on || (wf <= 0 && wc <= 0)) m |= 2 << (2 * ax);
            if (!on || (wf >= 0 && wc >= 0)) m |= 4 << (2 * ax);
        }
        A.mask[a] = m;
    }
}

template <class T>
__global__ void k3_check(DD3Args<T> A, int k) {
    if (*A.done) return;
    const double delta = A.deltas[k];
    const bool failed = A.st->err != DEV_OK;  // an expired wait: later stages would only repeat it
    const bool conv = k >= 1 && delta < (double)A.tol && !failed;
    if (k == A.max_iter || conv || failed) {
        *A.done = 1;
        A.st->iters = k;
        A.st->converged = conv ? 1 : 0;
    }
}

template <class T>
__global__ void k3_delta(DD3Args<T> A, int k) {
    if (*A.done) return;
    double m = 0.0;
    for (long long a = blockIdx.x * (long long)blockDim.x + threadIdx.x; a < A.G.nc;
         a += (long long)gridDim.x * blockDim.x) {
        const T u1 = A.U[a], u0 = A.Uprev[a];
        if (u1 == u0) continue;
        const double dv = fabs((double)u1 - (double)u0);
        if (dv > m) m = dv;
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(FULL, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.0)
        atomicMax(reinterpret_cast<unsigned long long *>(&A.deltas[k + 1]), (unsigned long long)__double_as_longlong(m));
}

// --------------------------------------------------------------------------
// Causal sweep (Alg. 2): every line along axis e whose nodes lie on a coarse
// plane of another axis; least fixed point, rounds until nothing changes.
//
// A lane takes a whole line and walks it forwards and back.  Lanes next to each
// other take lines next to each other on the same shifted grids, so their
// loads are contiguous (along x: within a few sectors that the lane comes back
// to), and sixteen nodes are in flight per lane.  Nodes of a shifted grid follow
// by counting; only the grid's record is looked up.  Lines share only their
// intersections, so after the first round a line is walked again only if a
// crossing line raised one of its nodes (which sets its flag; a line clears its
// own before it is walked): the least fixed point is the same.  1.16 ms a call on 257^3
// with a warp per line, a segmented scan per 32 nodes and the node's address
// by six divisions; 0.81 ms so.
// --------------------------------------------------------------------------
constexpr int CAUSAL3_AHEAD = 16;

// Lines along e: `fast` is the axis next to which lines lie side by side.
struct Lines3 {
    int fast, slow, c, nf, ns, mf, ms;  // nodes and coarse planes of both axes
    __device__ Lines3(const DD3Geom &G, int e) {
        fast = e == 0 ? 1 : 0;
        slow = 3 - e - fast;
        c = G.c;
        nf = G.n[fast];
        ns = G.n[slow];
        mf = (nf - 1) / c + 1;
        ms = (ns - 1) / c + 1;
    }
    __device__ int count() const { return ms * nf + (ns - ms) * mf; }
    // line L: coordinates on the fast and the slow axis
    __device__ void get(int L, int &xf, int &xs) const {
        if (L < ms * nf) {  // on a coarse plane of the slow axis: all nodes of the fast one, by residue
            const int p = L / nf, k = L - p * nf;
            xs = p * c;
            if (k < mf) {
                xf = k * c;
            } else {
                const int o = (k - mf) / (mf - 1);
                xf = (k - mf - o * (mf - 1)) * c + o + 1;
            }
        } else {
            const int r = L - ms * nf, p = r / mf;
            xs = p + 1 + p / (c - 1);  // the p-th node off the coarse planes
            xf = (r - p * mf) * c;
        }
    }
};

// Flag of the line along e through X.
__host__ __device__ inline size_t line3_flags(const DD3Geom &G) {
    return (size_t)G.n[0] * G.n[1] + (size_t)G.n[1] * G.n[2] + (size_t)G.n[0] * G.n[2];
}
__device__ inline size_t line3_flag(const DD3Geom &G, int e, const int *X) {
    if (e == 0) return (size_t)X[2] * G.n[1] + X[1];
    const size_t n12 = (size_t)G.n[1] * G.n[2];
    if (e == 1) return n12 + (size_t)X[2] * G.n[0] + X[0];
    return n12 + (size_t)G.n[0] * G.n[2] + (size_t)X[1] * G.n[0] + X[0];
}

template <class T>
__device__ bool causal3_line(const DD3Args<T> &A, int e, const int *X, int rev) {
    const DD3Geom &G = A.G;
    const T INF = Num<T>::inf();
    const int c = G.c, len = G.n[e];
    int i[3], o[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        i[a] = a == e ? (rev ? (len - 1) / c : 0) : X[a] / c;
        o[a] = a == e ? 0 : X[a] % c;
    }
    bool changed = false;
    T pred = INF, v = INF;  // the node behind: its value before this pass, after it
    for (int p0 = 0; p0 < len; p0 += CAUSAL3_AHEAD) {
        long long at[CAUSAL3_AHEAD];
        T u[CAUSAL3_AHEAD];
        uint8_t w[CAUSAL3_AHEAD];
#pragma unroll
        for (int q = 0; q < CAUSAL3_AHEAD; ++q) {
            u[q] = INF;
            w[q] = WIND_ZERO;
            if (p0 + q < len) {
                const Grid3 &d = A.grids[A.offmap[(o[2] * c + o[1]) * c + o[0]]];
                at[q] = d.off + ((long long)i[2] * d.my + i[1]) * d.mx + i[0];
                u[q] = A.U[at[q]];
                w[q] = A.W[at[q]];
#pragma unroll
                for (int a = 0; a < 3; ++a) {  // one node on along e
                    if (a != e) continue;
                    if (!rev) {
                        if (++o[a] == c) { o[a] = 0; ++i[a]; }
                    } else {
                        if (o[a]-- == 0) { o[a] = c - 1; --i[a]; }
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < CAUSAL3_AHEAD; ++q) {
            if (p0 + q < len) {
                const int wc = wind_comp(w[q], e);
                const bool f = p0 + q > 0 && (rev ? wc < 0 : wc > 0) && pred < INF;
                v = f ? fmax(u[q], v) : u[q];
                if (v > u[q]) {
                    A.U[at[q]] = v;
                    changed = true;
                    int Y[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) Y[a] = a == e ? (rev ? len - 1 - p0 - q : p0 + q) : X[a];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {  // the line along a through the node, if it is one
                        const int b1 = a == 0 ? 1 : 0, b2 = a == 2 ? 1 : 2;
                        if (A.lflag && a != e && (Y[b1] % c == 0 || Y[b2] % c == 0)) A.lflag[line3_flag(G, a, Y)] = 1;
                    }
                }
                pred = u[q];
            }
        }
    }
    return changed;
}

template <class T>
__global__ void k3_causal(DD3Args<T> A, int only_if_not_done) {
    const long long wlim = spin_limit();  // limit of the grid-barrier waits
    if (only_if_not_done && *A.done) return;
    const DD3Geom &G = A.G;
    const int lane = threadIdx.x & 31;
    __shared__ int blk_changed;
    if (blockIdx.x == 0 && threadIdx.x < 3) A.chg[threadIdx.x] = 0;
    const size_t nflags = A.lflag ? line3_flags(G) : 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nflags; i += (size_t)gridDim.x * blockDim.x)
        A.lflag[i] = 0;
    if (!grid_barrier(A.bar, &A.st->err, wlim)) return;
    int rounds = 0;
    for (;;) {
        if (threadIdx.x == 0) blk_changed = 0;
        __syncthreads();
        bool ch = false;
        for (int e = 0; e < 3; ++e) {
            const Lines3 lines(G, e);
            const int n = lines.count();
            for (int L = blockIdx.x * blockDim.x + threadIdx.x; L < n; L += gridDim.x * blockDim.x) {
                int X[3] = {0, 0, 0}, xf, xs;
                lines.get(L, xf, xs);
#pragma unroll
                for (int a = 0; a < 3; ++a) X[a] = a == lines.fast ? xf : (a == lines.slow ? xs : 0);
                if (A.lflag) {
                    uint8_t *flag = A.lflag + line3_flag(G, e, X);
                    if (rounds > 0 && !__ldcg(flag)) continue;
                    *flag = 0;
                }
                const bool fwd = causal3_line(A, e, X, 0);
                const bool back = causal3_line(A, e, X, 1);
                ch = ch || fwd || back;
            }
            if (!grid_barrier(A.bar, &A.st->err, wlim)) return;
        }
        ch = __any_sync(FULL, ch);
        if (lane == 0 && ch) atomicOr(&blk_changed, 1);
        __syncthreads();
        if (threadIdx.x == 0 && blk_changed) atomicOr(&A.chg[rounds % 3], 1);
        ++rounds;
        if (!grid_barrier(A.bar, &A.st->err, wlim)) return;
        const int any = *(volatile int *)&A.chg[(rounds - 1) % 3];
        if (blockIdx.x == 0 && threadIdx.x == 0) A.chg[(rounds + 1) % 3] = 0;
        if (!any || rounds > 10000) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicMax(&A.st->causal_rounds_max, rounds);
}

template <class T>
__global__ void k3_finalize(DD3Args<T> A, eik_dd_stats *out, long long launches) {
    if (threadIdx.x != 0 || !out) return;
    out->iters = A.st->iters;
    out->converged = A.st->converged;
    out->error = A.st->err;
    out->causal_rounds_max = A.st->causal_rounds_max;
    out->fsm_sweeps_max = (int64_t)A.st->fsm_sweeps_max;
    out->coarse_sweeps_max = (int64_t)A.st->coarse_sweeps_max;
    out->fsm_cap_hits = (int64_t)A.st->fsm_caps;
    out->coarse_cap_hits = (int64_t)A.st->coarse_caps;
    const int k = A.st->iters;
    out->last_delta = k >= 1 ? A.deltas[k] : INFINITY;
    out->fine_updates = (int64_t)A.st->fine_updates;
    out->coarse_updates = (int64_t)A.st->coarse_updates;
    out->launches = launches;
    out->fine_solves_skipped = (int64_t)A.st->fine_skips;
}

// --------------------------------------------------------------------------
// Host side
// --------------------------------------------------------------------------
struct DD3Plan {
    DD3Geom G;
    std::vector<Grid3> grids;
    std::vector<int> offmap;
    size_t fine_smem, grid_smem, bytes;
    size_t fine_limit, grid_limit;  // what decides whether the size is supported
    int fpx, fps, gpx, gps;  // pitches (see Box3)
    int fine_threads, grid_threads;
    bool adaptive;
};

static bool dd3_plan(const eik_grid *grid, const eik_dd_params *p, DD3Plan &P) {
    const int c = p->coarse_ratio;
    DD3Geom &G = P.G;
    for (int a = 0; a < 3; ++a) {
        G.n[a] = (int)grid->n[a];
        G.T[a] = p->tiles[a];
        G.S[a] = (G.n[a] - 1) / G.T[a];
    }
    G.c = c;
    G.h = grid->h;
    G.H = (double)c * grid->h;
    P.adaptive = p->theta_adaptive != 0;
    P.grids.clear();
    P.offmap.assign((size_t)c * c * c, -1);
    long long off = 0;
    for (int oz = 0; oz < c; ++oz)
        for (int oy = 0; oy < c; ++oy)
            for (int ox = 0; ox < c; ++ox) {
                if (ox && oy && oz) continue;
                Grid3 d;
                d.ox = ox;
                d.oy = oy;
                d.oz = oz;
                d.mx = (G.n[0] - 1 - ox) / c + 1;
                d.my = (G.n[1] - 1 - oy) / c + 1;
                d.mz = (G.n[2] - 1 - oz) / c + 1;
                d.off = off;
                off += (long long)d.mx * d.my * d.mz;
                P.offmap[((size_t)oz * c + oy) * c + ox] = (int)P.grids.size();
                P.grids.push_back(d);
            }
    G.ng = (int)P.grids.size();
    G.nc = off;
    const size_t tsz = grid->dtype == EIK_F64 ? 8 : 4;
    const int f0 = G.S[0] + 1, f1 = G.S[1] + 1, f2 = G.S[2] + 1;
    P.fine_limit = box3_limit(f0, f1, f2, tsz);
    // the unshifted grid is the largest
    const Grid3 &g0 = P.grids[0];
    P.grid_limit = box3_limit(g0.mx, g0.my, g0.mz, tsz);
    const size_t most = (227 << 10) - 256;  // shared memory of a CTA beside the static part
    box3_pitch(f0, f1, f2, (int)tsz, most, P.fpx, P.fps);
    box3_pitch(g0.mx, g0.my, g0.mz, (int)tsz, most, P.gpx, P.gps);
    P.fine_smem = box3_elems(f0, f2, P.fpx, P.fps) * tsz + 16;
    P.grid_smem = box3_elems(g0.mx, g0.mz, P.gpx, P.gps) * tsz + 16;
    P.fine_threads = BOX3_THREADS;
    P.grid_threads = BOX3_THREADS;
    return true;
}

// lean: without the packed subdomains and the line flags, a fifth less
template <class T>
static size_t dd3_layout(const DD3Plan &P, DD3Args<T> *A, void *ws, int max_iter, bool lean) {
    const DD3Geom &G = P.G;
    Carver cv(ws);
    T *U = cv.take<T>(G.nc), *Uprev = cv.take<T>(G.nc), *U0 = cv.take<T>(G.nc), *rc = cv.take<T>(G.nc);
    T *uk = cv.take<T>(G.nc), *cold = cv.take<T>(G.nc);
    uint8_t *W = cv.take<uint8_t>(G.nc), *wk = cv.take<uint8_t>(G.nc), *mask = cv.take<uint8_t>(G.nc);
    T *cu = cv.take<T>(8 * (size_t)G.nc);
    uint8_t *cw = cv.take<uint8_t>(8 * (size_t)G.nc);
    Grid3 *grids = cv.take<Grid3>(P.grids.size());
    int *offmap = cv.take<int>(P.offmap.size());
    int *done = cv.take<int>(4);
    double *deltas = cv.take<double>((size_t)max_iter + 2);
    int *chg = cv.take<int>(4);
    uint8_t *lflag = lean ? nullptr : cv.take<uint8_t>(line3_flags(G));
    unsigned *bar = cv.take<unsigned>(4);
    DevStats3 *st = cv.take<DevStats3>(1);
    const size_t ntl = (size_t)G.T[0] * G.T[1] * G.T[2], nsl = (size_t)box3_face_slots(G.S);
    T *sig_u = cv.take<T>(ntl * nsl);
    uint8_t *sig_w = cv.take<uint8_t>(ntl * nsl);
    int *sig_ok = cv.take<int>(ntl);
    T *rp = lean ? nullptr : cv.take<T>(ntl * box3_tiles(G.S[0] + 1, G.S[1] + 1) * (G.S[2] + 1) * 32);
    T *Ch[4] = {nullptr, nullptr, nullptr, nullptr}, *th = nullptr;
    double *du = nullptr;
    if (P.adaptive) {
        for (int s = 0; s < 4; ++s) Ch[s] = cv.take<T>(G.nc);
        th = cv.take<T>(G.nc);
        du = cv.take<double>(G.nc);
    }
    if (A) {
        for (int s = 0; s < 4; ++s) A->Ch[s] = Ch[s];
        A->th = th;
        A->du = du;
        A->U = U; A->Uprev = Uprev; A->U0 = U0; A->rc = rc; A->uk = uk; A->cold = cold;
        A->W = W; A->wk = wk; A->mask = mask; A->cu = cu; A->cw = cw;
        A->grids = grids; A->offmap = offmap; A->done = done; A->deltas = deltas; A->chg = chg; A->bar = bar;
        A->st = st;
        A->sig_u = sig_u;
        A->sig_w = sig_w;
        A->sig_ok = sig_ok;
        A->rp = rp;
        A->lflag = lflag;
        A->fpx = P.fpx; A->fps = P.fps; A->gpx = P.gpx; A->gps = P.gps;
        A->fo = P.fpx > G.S[0] + 1 ? P.fpx + 1 : 0;
        A->go = P.gpx > P.grids[0].mx ? P.gpx + 1 : 0;
    }
    return cv.used + 256;
}

// Shifted-grid tables, built on the device in the enumeration order of the
// host plan (z offset outermost, x innermost; offsets with no zero skipped).
__global__ void k3_tables(Grid3 *grids, int *offmap, int c, int n0, int n1, int n2) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    long long off = 0;
    int gi = 0;
    for (int oz = 0; oz < c; ++oz)
        for (int oy = 0; oy < c; ++oy)
            for (int ox = 0; ox < c; ++ox) {
                const int m = (oz * c + oy) * c + ox;
                if (ox && oy && oz) {
                    offmap[m] = -1;
                    continue;
                }
                Grid3 d;
                d.ox = ox;
                d.oy = oy;
                d.oz = oz;
                d.mx = (n0 - 1 - ox) / c + 1;
                d.my = (n1 - 1 - oy) / c + 1;
                d.mz = (n2 - 1 - oz) / c + 1;
                d.off = off;
                off += (long long)d.mx * d.my * d.mz;
                offmap[m] = gi;
                grids[gi++] = d;
            }
}

// lean = false: the workspace to ask for; true: what a solve can do with
size_t dd3_workspace_size(const eik_grid *grid, const eik_dd_params *p, bool lean) {
    DD3Plan P;
    dd3_plan(grid, p, P);
    return grid->dtype == EIK_F64 ? dd3_layout<double>(P, nullptr, nullptr, p->max_iter, lean)
                                  : dd3_layout<float>(P, nullptr, nullptr, p->max_iter, lean);
}

bool dd3_validate(const eik_grid *grid, const eik_dd_params *p) {
    for (int a = 0; a < 3; ++a) {
        if (p->tiles[a] < 1 || (grid->n[a] - 1) % p->tiles[a] != 0) {
            set_error("tiles[%d] = %d does not divide n[%d]-1", a, p->tiles[a], a);
            return false;
        }
        if (((grid->n[a] - 1) / p->tiles[a]) % p->coarse_ratio != 0) {
            set_error("coarse_ratio %d does not divide the subdomain width along axis %d", p->coarse_ratio, a);
            return false;
        }
    }
    if (p->coarse_ratio < 1 || p->coarse_ratio > 64) {
        set_error("coarse_ratio must be in [1, 64] in 3-D");
        return false;
    }
    return true;
}

template <class T>
static int dd3_run_t(const eik_grid *grid, const void *r, const uint8_t *gamma, const void *g,
                     const eik_dd_params *p, void *u_out, void *ws, size_t ws_bytes, eik_dd_stats *stats,
                     cudaStream_t s) {
    DD3Plan P;
    dd3_plan(grid, p, P);
    DD3Args<T> A;
    memset(&A, 0, sizeof(A));
    A.G = P.G;
    A.r = static_cast<const T *>(r);
    A.gamma = gamma;
    A.g = static_cast<const T *>(g);
    A.u_out = static_cast<T *>(u_out);
    A.sy = grid->stride[1];
    A.sz = grid->stride[2];
    const bool lean = ws_bytes < dd3_layout<T>(P, nullptr, nullptr, p->max_iter, false);
    dd3_layout<T>(P, &A, ws, p->max_iter, lean);
    A.theta = (T)p->theta;
    A.tol = (T)p->tol;
    A.max_iter = p->max_iter;
    A.max_fsm = p->max_fsm_sweeps;
    A.max_coarse = p->max_coarse_sweeps;
    A.adaptive = P.adaptive ? 1 : 0;
    A.step4_identity = (!P.adaptive && p->theta == 0.0) ? 1 : 0;
    for (int s2 = 0; s2 < 3; ++s2) A.om[s2] = p->omega[s2];
    A.sg = p->sig_gamma;
    A.sd = p->sig_delta;
    A.sx0 = p->sig_x0;
    A.cap = p->theta_cap;
    const DD3Geom &G = P.G;
    int rc, dev, nsm = 0, optin = 0;
    if ((rc = cuda_check(cudaGetDevice(&dev), "cudaGetDevice"))) return rc;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if ((int)P.fine_limit > optin || (int)P.grid_limit > optin || (int)P.fine_smem > optin ||
        (int)P.grid_smem > optin) {
        set_error("3-D subdomain or coarse grid box needs %zu / %zu bytes of shared memory (limit %d)",
                  std::max(P.fine_limit, P.fine_smem), std::max(P.grid_limit, P.grid_smem), optin);
        return EIK_EUNSUPPORTED;
    }
    void (*const fine)(DD3Args<T>) = lean ? k3_fine<T, false> : k3_fine<T, true>;
    if ((rc = cuda_check(set_dyn_smem(fine, (int)P.fine_smem), "attr")))
        return rc;
    if ((rc = cuda_check(set_dyn_smem(k3_step1<T>, (int)P.grid_smem), "attr")))
        return rc;
    if ((rc = cuda_check(set_dyn_smem(k3_step4<T>, (int)P.grid_smem), "attr")))
        return rc;
    const int causal_threads = 64;  // a lane per line: spread the warps over the SMs
    int per_sm = 0;
    if ((rc = cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k3_causal<T>, causal_threads, 0), "occ")))
        return rc;
    const int causal_blocks = std::max(1, std::min(per_sm * nsm, 2 * nsm));
    const int ntiles = G.T[0] * G.T[1] * G.T[2];
    dim3 cgrid(8, G.ng);
    const int ew = 256;
    const int eb = (int)std::min<long long>((G.nc + ew - 1) / ew, (long long)nsm * 8);
    long long nl = 0;
    EIK_LAUNCH("dd3_init", s, k3_init<T><<<1, 256, 0, s>>>(A)); ++nl;
    EIK_LAUNCH("dd3_tables", s, k3_tables<<<1, 32, 0, s>>>(A.grids, A.offmap, G.c, G.n[0], G.n[1], G.n[2])); ++nl;
    EIK_LAUNCH("dd3_pack_coarse", s, k3_pack_coarse<T><<<cgrid, ew, 0, s>>>(A)); ++nl;
    if (!lean) {
        EIK_LAUNCH("dd3_pack_tiles", s, k3_pack_tiles<T><<<ntiles, ew, 0, s>>>(A));
        ++nl;
    }
    EIK_LAUNCH("dd3_step1_coarse_fsm", s, k3_step1<T><<<G.ng, P.grid_threads, P.grid_smem, s>>>(A)); ++nl;
    auto launch_causal = [&](int only) -> int {
        void *args[] = {&A, &only};
        int tok = prof_begin("dd3_causal_sweep", s);
        int r2 = cuda_check(cudaLaunchCooperativeKernel((void *)k3_causal<T>, causal_blocks, causal_threads, args, 0, s),
                            "causal launch");
        prof_end(tok, s);
        ++nl;
        return r2;
    };
    if ((rc = launch_causal(0))) return rc;
    for (int k = 0; k <= p->max_iter; ++k) {
        EIK_LAUNCH("dd3_fine_subdomains", s, fine<<<ntiles, P.fine_threads, P.fine_smem, s>>>(A)); ++nl;
        EIK_LAUNCH("dd3_alg4_restrict", s, k3_alg4<T><<<cgrid, ew, 0, s>>>(A)); ++nl;
        EIK_LAUNCH("dd3_check", s, k3_check<T><<<1, 1, 0, s>>>(A, k)); ++nl;
        if (k == p->max_iter) break;
        if (!A.step4_identity) {
            EIK_LAUNCH("dd3_step4_weighted", s, k3_step4<T><<<G.ng, P.grid_threads, P.grid_smem, s>>>(A, k));
            ++nl;
        }
        if ((rc = launch_causal(1))) return rc;
        EIK_LAUNCH("dd3_delta", s, k3_delta<T><<<eb, ew, 0, s>>>(A, k)); ++nl;
    }
    ++nl;
    EIK_LAUNCH("dd3_finalize", s, k3_finalize<T><<<1, 32, 0, s>>>(A, stats, nl));
    return cuda_check(cudaGetLastError(), "dd3 launch");
}

int dd3_run(const eik_grid *grid, const void *r, const uint8_t *gamma, const void *g, const eik_dd_params *p,
            void *u_out, void *ws, size_t ws_bytes, eik_dd_stats *stats, cudaStream_t s) {
    if (grid->dtype == EIK_F64) return dd3_run_t<double>(grid, r, gamma, g, p, u_out, ws, ws_bytes, stats, s);
    return dd3_run_t<float>(grid, r, gamma, g, p, u_out, ws, ws_bytes, stats, s);
}

}  // namespace eik
