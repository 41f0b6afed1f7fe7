// eik_fsm.cu -- plain fast sweeping method on the whole grid (Sec. 1.1), the
// baseline the domain decomposition is compared against, plus the shared host
// helpers of the C ABI (error text, version).
//
// Sweeps cycle through the four orderings until one changes nothing.  Small grids
// are swept by one warp in shared memory, in one launch (box2.cuh).  Larger ones
// are one box for the warp-systolic engine, one warp per 32-column block: all
// blocks in one CTA up to MAX_SINGLE_NB, else spread over co-resident CTAs.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "box2.cuh"
#include "engine.cuh"
#include "host_util.h"
#include "prof.h"
#include "ptr_table.cuh"

#include <string>
#include <vector>

namespace eik {

EIK_SPIN_LIMIT_SETTER(set_spin_limit_fsm)

static thread_local char g_err[512];

// ---- optional per-launch event timing -------------------------------------
struct ProfRec {
    const char *name;
    cudaEvent_t a, b;
};
static bool g_prof_on = false;
static std::vector<ProfRec> g_prof;
static std::vector<cudaEvent_t> g_prof_pool;

static cudaEvent_t prof_event() {
    if (!g_prof_pool.empty()) {
        cudaEvent_t e = g_prof_pool.back();
        g_prof_pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

int prof_begin(const char *name, cudaStream_t s) {
    if (!g_prof_on) return -1;
    ProfRec r{name, prof_event(), prof_event()};
    cudaEventRecord(r.a, s);
    g_prof.push_back(r);
    return (int)g_prof.size() - 1;
}

void prof_end(int token, cudaStream_t s) {
    if (token < 0) return;
    cudaEventRecord(g_prof[token].b, s);
}

void set_error(const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

struct FsmDev {
    unsigned long long sweeps;
    int converged;
    int err;
};

template <class T>
struct FsmArgs {
    const T *r;
    const uint8_t *gamma;
    const T *g;
    T *u;
    long long sy;
    int nx, ny, nb, nstepp;
    T *state;
    T *rsk;
    T *ghands;   // multi-CTA hand-off columns [nb][hand_elems(ny)]
    int *gctl;   // multi-CTA control words
    FsmDev *dev;
    T h;
    long long max_sweeps;
    int launches;
    int multi;   // multi-CTA form
};

// Skewed slowness r h (NaN at positions
// outside the box and Gamma nodes), then the state (Sec. 1.1 initialisation:
// Gamma fixed at g, everything else large, padding columns included) and, for
// the multi-CTA form, the empty hand-off columns.
template <class T>
__device__ void fsm_pack_body(const FsmArgs<T> &A, size_t bid, size_t nbid) {
    skew_pack<T, 1>(A.rsk, 0, A.nx, A.ny, A.nb, A.nstepp, bid, nbid, Num<T>::nan(), [&](int, int x, int y) {
        const size_t gi = (size_t)y * A.sy + x;
        return FsmPolicy<T>::node(A.gamma[gi] != 0, A.r[gi], A.h);
    });
    const size_t total = (size_t)A.nb * A.ny * 32;
    for (size_t t = bid * blockDim.x + threadIdx.x; t < total; t += nbid * blockDim.x) {
        const size_t row = t >> 5;
        const int b = (int)(row / A.ny), y = (int)(row - (size_t)b * A.ny), x = 32 * b + (int)(t & 31);
        T v = Num<T>::inf();
        if (x < A.nx) {
            const size_t gi = (size_t)y * A.sy + x;
            if (A.gamma[gi]) v = gamma_value(A.g[gi]);
        }
        A.state[t] = v;
    }
    if (A.multi)
        for (size_t t = bid * blockDim.x + threadIdx.x; t < A.nb * hand_elems(A.ny); t += nbid * blockDim.x)
            A.ghands[t] = Hand<T>::empty();
}

template <class T>
__global__ void k_fsm_pack(FsmArgs<T> A) {
    fsm_pack_body(A, blockIdx.x, gridDim.x);
}

template <class T>
__device__ void fsm_run_body(const FsmArgs<T> &A, char *smem) {
    Box<T, 1> bx;
    bx.u = A.state;
    bx.st[0] = A.rsk;
    bx.sb = nullptr;
    bx.ny = A.ny;
    bx.nb = A.nb;
    bx.nstepp = A.nstepp;
    FsmPolicy<T> pol;
    long long sweeps;
    bool conv;
    if (threadIdx.x == 0) A.dev->err = 0;
    __syncthreads();
    engine_run<T, 1, false>(bx, pol, A.max_sweeps, smem, sweeps, conv, &A.dev->err);
    if (threadIdx.x == 0) {
        A.dev->sweeps = (unsigned long long)sweeps;
        A.dev->converged = conv ? 1 : 0;
    }
}

template <class T>
__global__ void __maxnreg__((RegCap<T, 112, 160>::v)) k_fsm_run(FsmArgs<T> A) {
    extern __shared__ __align__(16) char smem[];
    fsm_run_body(A, smem);
}

// Multi-CTA form for grids wider than one CTA's blocks: cooperative launch,
// hand-offs and control words in global memory.
template <class T>
__global__ void k_fsm_init_global(FsmArgs<T> A) {
    engine_global_init(A.gctl, A.nb);
    if (threadIdx.x == 0) A.dev->err = 0;
}

template <class T>
__device__ void fsm_run_global_body(const FsmArgs<T> &A, char *smem, int cta) {
    Box<T, 1> bx;
    bx.u = A.state;
    bx.st[0] = A.rsk;
    bx.sb = nullptr;
    bx.ny = A.ny;
    bx.nb = A.nb;
    bx.nstepp = A.nstepp;
    FsmPolicy<T> pol;
    long long sweeps;
    bool conv;
    engine_run<T, 1, false, true>(bx, pol, A.max_sweeps, smem, sweeps, conv, &A.dev->err, A.ghands, A.gctl, cta);
}

template <class T>
__global__ void __maxnreg__((RegCap<T, 112, 160>::v)) k_fsm_run_global(FsmArgs<T> A) {
    extern __shared__ __align__(16) char smem[];
    fsm_run_global_body(A, smem, (int)blockIdx.x);
}

template <class T>
__device__ void fsm_unpack_body(const FsmArgs<T> &A, eik_fsm_stats *out, size_t bid, size_t nbid) {
    const size_t total = (size_t)A.nx * A.ny;
    for (size_t t = bid * blockDim.x + threadIdx.x; t < total; t += nbid * blockDim.x) {
        int x = (int)(t % A.nx), y = (int)(t / A.nx);
        A.u[(size_t)y * A.sy + x] = A.state[box_index(x, y, A.ny)];
    }
    if (out && bid == 0 && threadIdx.x == 0) {
        long long sweeps = (long long)A.dev->sweeps;
        bool conv = A.dev->converged != 0;
        if (A.multi) engine_result(A.gctl, A.max_sweeps, sweeps, conv);
        out->sweeps = sweeps;
        out->converged = conv ? 1 : 0;
        out->error = A.dev->err;
        out->updates = sweeps * A.nx * A.ny;
        out->launches = A.launches;
    }
}

template <class T>
__global__ void k_fsm_unpack(FsmArgs<T> A, eik_fsm_stats *out) {
    fsm_unpack_body(A, out, blockIdx.x, gridDim.x);
}

// A small grid from the caller's arrays to u in one launch, swept by one warp in
// shared memory (box2.cuh).  97 x 101 FP32, 24 sweeps: 0.45 ms a call, packed and
// by the engine 0.67 ms.
template <int K, class T>
__device__ __forceinline__ void fsm_box_body(const FsmArgs<T> &A, char *smem, eik_fsm_stats *out) {
    const Box2<K> B(A.nx, A.ny);
    T *const su = reinterpret_cast<T *>(smem), *const sr = su + B.cells();
    B.clear(su, sr);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int y = warp; y < A.ny; y += nw)
        for (int x = lane; x < A.nx; x += 32) {
            const size_t gi = (size_t)y * A.sy + x;
            const bool gam = A.gamma[gi] != 0;
            const int q = B.at(x, y);
            sr[q] = FsmPolicy<T>::node(gam, A.r[gi], A.h);
            if (gam) su[q] = box2_gamma(A.g[gi]);
        }
    __syncthreads();
    if (warp == 0) {
        long long sweeps;
        bool conv;
        box2_sweeps<K, T>(B, (unsigned)__cvta_generic_to_shared(su), (unsigned)__cvta_generic_to_shared(sr),
                          A.max_sweeps, sweeps, conv);
        if (out && lane == 0) {
            out->sweeps = sweeps;
            out->converged = conv ? 1 : 0;
            out->error = DEV_OK;
            out->updates = sweeps * A.nx * A.ny;
            out->launches = A.launches;
        }
    }
    __syncthreads();
    for (int y = warp; y < A.ny; y += nw)
        for (int x = lane; x < A.nx; x += 32) A.u[(size_t)y * A.sy + x] = su[B.at(x, y)];
}

constexpr int FSM_BOX_THREADS = 512;  // for the copies in and out

template <int K, class T>
__global__ void __launch_bounds__(FSM_BOX_THREADS) k_fsm_box(FsmArgs<T> A, eik_fsm_stats *out) {
    extern __shared__ __align__(16) char smem[];
    fsm_box_body<K, T>(A, smem, out);
}
template <class T>
constexpr void (*fsm_box_kernel(int k))(FsmArgs<T>, eik_fsm_stats *) {
    if constexpr (box2_kmax<T>() > 2)
        if (k > 2) return k == 3 ? k_fsm_box<3, T> : k_fsm_box<4, T>;
    return k == 1 ? k_fsm_box<1, T> : k_fsm_box<2, T>;
}

// Widest grid (32-column blocks) swept by one CTA.  Above it the blocks' warps
// share too few schedulers and spreading them over CTAs wins in spite of the
// slower hand-off, which counts most where a grid has few rows.  ms a solve, one
// CTA / several: FP32 257^2 3.55 / 3.36 and 20 x 257 1.74 / 1.92, 289^2 4.27 / 4.10
// and 20 x 289 2.07 / 2.24, 353^2 6.15 / 5.48 and 20 x 353 2.99 / 2.82; FP64 161^2
// 8.72 / 8.99, 257^2 21.5 / 20.1 and 20 x 280 9.88 / 10.3.
constexpr int MAX_SINGLE_NB = 9;

struct FsmPlan {
    int nx, ny, nb, nstepp;
    size_t smem, bytes;
    size_t gsmem;  // multi-CTA shared memory per CTA
    int wpc;       // multi-CTA warps (blocks) per CTA
};

template <class T>
static size_t fsm_layout(const FsmPlan &P, FsmArgs<T> *A, void *ws) {
    Carver cv(ws);
    T *state = cv.take<T>((size_t)P.nb * P.ny * 32);
    T *rsk = cv.take<T>((size_t)4 * P.nb * P.nstepp * 32);
    T *ghands = cv.take<T>(P.nb * hand_elems(P.ny));
    int *gctl = cv.take<int>(engine_global_ints(P.nb));
    FsmDev *dev = cv.take<FsmDev>(1);
    if (A) {
        A->state = state;
        A->rsk = rsk;
        A->ghands = ghands;
        A->gctl = gctl;
        A->dev = dev;
    }
    return cv.used + 256;
}

static bool fsm_plan(const eik_grid *grid, FsmPlan &P) {
    if (!valid_grid_common(grid, 2)) return false;
    P.nx = (int)grid->n[0];
    P.ny = (int)grid->n[1];
    P.nb = ceil32(P.nx);
    P.nstepp = nstep_whole_grid(P.ny);
    P.smem = grid->dtype == EIK_F64 ? engine_smem_bytes<double, 1, false>(P.nb, P.ny)
                                     : engine_smem_bytes<float, 1, false>(P.nb, P.ny);
    // FP64: one warp per CTA, each with an SM's FP64 pipe of its own (two warps
    // share it: 1401 x 701 FP64 1119 us a sweep, one 1073); FP32: 1 to 4 are alike
    P.wpc = grid->dtype == EIK_F64 ? 1 : 2;
    P.gsmem = grid->dtype == EIK_F64 ? engine_smem_bytes<double, 1, false, true>(P.wpc, P.ny)
                                      : engine_smem_bytes<float, 1, false, true>(P.wpc, P.ny);
    P.bytes = grid->dtype == EIK_F64 ? fsm_layout<double>(P, nullptr, nullptr) : fsm_layout<float>(P, nullptr, nullptr);
    return true;
}

template <class T>
static int fsm_run(const eik_grid *grid, const FsmPlan &P, const void *r, const uint8_t *gamma, const void *g,
                   void *u, int64_t max_sweeps, void *ws, eik_fsm_stats *stats, cudaStream_t s) {
    FsmArgs<T> A;
    memset(&A, 0, sizeof(A));
    A.r = static_cast<const T *>(r);
    A.gamma = gamma;
    A.g = static_cast<const T *>(g);
    A.u = static_cast<T *>(u);
    A.sy = grid->stride[1];
    A.nx = P.nx;
    A.ny = P.ny;
    A.nb = P.nb;
    A.nstepp = P.nstepp;
    A.h = (T)grid->h;
    A.max_sweeps = max_sweeps;
    fsm_layout<T>(P, &A, ws);
    int rc;
    // one problem, one CTA: it may take most of an SM's shared memory
    if (const int k = box2_use<T>(P.nx, P.ny, 200 << 10)) {
        A.launches = 1;
        const size_t smem = box2_smem_bytes<T>(P.nx, P.ny);
        void (*const kernel)(FsmArgs<T>, eik_fsm_stats *) = fsm_box_kernel<T>(k);
        if ((rc = cuda_check(set_dyn_smem(kernel, (int)smem), "smem attr"))) return rc;
        EIK_LAUNCH("fsm_sweeps", s, kernel<<<1, FSM_BOX_THREADS, smem, s>>>(A, stats));
        return cuda_check(cudaGetLastError(), "fsm launch");
    }
    int dev, optin = 0, nsm = 0;
    if ((rc = cuda_check(cudaGetDevice(&dev), "cudaGetDevice"))) return rc;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncAttributes fa;
    if ((rc = cuda_check(cudaFuncGetAttributes(&fa, k_fsm_run<T>), "func attr"))) return rc;
    const bool single = (int)P.smem <= optin && P.nb <= MAX_SINGLE_NB && regs_fit(fa, P.nb);
    A.launches = single ? 3 : 4;
    A.multi = single ? 0 : 1;
    const size_t total = (size_t)P.nx * P.ny;
    const int tb = (int)std::min<size_t>((total + 255) / 256, (size_t)nsm * 16);
    EIK_LAUNCH("fsm_pack", s, k_fsm_pack<T><<<tb, 256, 0, s>>>(A));
    if (single) {
        if ((rc = cuda_check(set_dyn_smem(k_fsm_run<T>, (int)P.smem), "smem attr")))
            return rc;
        EIK_LAUNCH("fsm_sweeps", s, k_fsm_run<T><<<1, 32 * P.nb, P.smem, s>>>(A));
    } else {
        // one CTA per P.wpc blocks, all co-resident
        const int nblk = (P.nb + P.wpc - 1) / P.wpc;
        if ((rc = cuda_check(set_dyn_smem(k_fsm_run_global<T>, (int)P.gsmem), "smem attr")))
            return rc;
        int per_sm = 0;
        if ((rc = cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fsm_run_global<T>, 32 * P.wpc,
                                                                          P.gsmem), "occupancy")))
            return rc;
        if (per_sm * nsm < nblk) {
            set_error("grid of %d x %d nodes needs %d co-resident CTAs, the device holds %d", P.nx, P.ny, nblk,
                      per_sm * nsm);
            return EIK_EUNSUPPORTED;
        }
        EIK_LAUNCH("fsm_init", s, k_fsm_init_global<T><<<1, 256, 0, s>>>(A));
        void *args[] = {&A};
        int tok = prof_begin("fsm_sweeps", s);
        rc = cuda_check(cudaLaunchCooperativeKernel((void *)k_fsm_run_global<T>, nblk, 32 * P.wpc, args, P.gsmem, s),
                        "fsm cooperative launch");
        prof_end(tok, s);
        if (rc) return rc;
    }
    EIK_LAUNCH("fsm_unpack", s, k_fsm_unpack<T><<<tb, 256, 0, s>>>(A, stats));
    return cuda_check(cudaGetLastError(), "fsm launch");
}


// --------------------------------------------------------------------------
// Many right-hand sides (sources Gamma_p, boundary values g_p) on one grid and
// one slowness: the per-problem kernels of fsm_run, each launch covering every
// problem (the multi-CTA sweep form in co-resident groups of problems).
// --------------------------------------------------------------------------
template <class T>
struct FsmMany {
    FsmArgs<T> A;            // shared fields; the per-problem ones are set by fsm_prob
    const void *const *tab;  // [3][nprob]: gamma, g, u
    char *ws0;               // workspace of problem 0; problem p at ws0 + p * per
    size_t per;
    size_t o_state, o_rsk, o_ghands, o_gctl, o_dev;  // offsets inside a problem's region
    int nprob;
};

template <class T>
__device__ __forceinline__ FsmArgs<T> fsm_prob(const FsmMany<T> &M, int p) {
    FsmArgs<T> A = M.A;
    A.gamma = static_cast<const uint8_t *>(M.tab[p]);
    A.g = static_cast<const T *>(M.tab[M.nprob + p]);
    A.u = static_cast<T *>(const_cast<void *>(M.tab[2 * M.nprob + p]));
    char *b = M.ws0 + (size_t)p * M.per;
    A.state = reinterpret_cast<T *>(b + M.o_state);
    A.rsk = reinterpret_cast<T *>(b + M.o_rsk);
    A.ghands = reinterpret_cast<T *>(b + M.o_ghands);
    A.gctl = reinterpret_cast<int *>(b + M.o_gctl);
    A.dev = reinterpret_cast<FsmDev *>(b + M.o_dev);
    return A;
}

template <class T>
__global__ void k_fsmm_pack(FsmMany<T> M) {
    fsm_pack_body(fsm_prob(M, blockIdx.y), blockIdx.x, gridDim.x);
}

template <class T>
__global__ void __maxnreg__((RegCap<T, 112, 160>::v)) k_fsmm_run(FsmMany<T> M) {
    extern __shared__ __align__(16) char smem[];
    fsm_run_body(fsm_prob(M, blockIdx.x), smem);
}

template <class T>
__global__ void k_fsmm_init_global(FsmMany<T> M) {
    const FsmArgs<T> A = fsm_prob(M, blockIdx.x);
    engine_global_init(A.gctl, A.nb);
    if (threadIdx.x == 0) A.dev->err = 0;
}

// CTA c of the launch serves problem p0 + c / nblk as its CTA c % nblk
template <class T>
__global__ void __maxnreg__((RegCap<T, 112, 160>::v)) k_fsmm_run_global(FsmMany<T> M, int p0, int nblk) {
    extern __shared__ __align__(16) char smem[];
    fsm_run_global_body(fsm_prob(M, p0 + (int)blockIdx.x / nblk), smem, (int)blockIdx.x % nblk);
}

template <class T>
__global__ void k_fsmm_unpack(FsmMany<T> M, eik_fsm_stats *out) {
    fsm_unpack_body(fsm_prob(M, blockIdx.y), out ? out + blockIdx.y : nullptr, blockIdx.x, gridDim.x);
}

template <int K, class T>
__global__ void __launch_bounds__(FSM_BOX_THREADS) k_fsmm_box(FsmMany<T> M, eik_fsm_stats *out) {
    extern __shared__ __align__(16) char smem[];
    fsm_box_body<K, T>(fsm_prob(M, blockIdx.x), smem, out ? out + blockIdx.x : nullptr);
}
template <class T>
constexpr void (*fsmm_box_kernel(int k))(FsmMany<T>, eik_fsm_stats *) {
    if constexpr (box2_kmax<T>() > 2)
        if (k > 2) return k == 3 ? k_fsmm_box<3, T> : k_fsmm_box<4, T>;
    return k == 1 ? k_fsmm_box<1, T> : k_fsmm_box<2, T>;
}

struct FsmManyPlan {
    FsmPlan P;
    size_t tab_bytes, per, bytes;
};

static bool fsm_many_plan(const eik_grid *grid, int nprob, FsmManyPlan &M) {
    if (nprob < 1 || nprob > 65535) {
        set_error("nprob = %d out of range [1, 65535]", nprob);
        return false;
    }
    if (!fsm_plan(grid, M.P)) return false;
    M.tab_bytes = ((size_t)3 * nprob * sizeof(void *) + 255) & ~(size_t)255;
    M.per = (M.P.bytes + 255) & ~(size_t)255;
    M.bytes = M.tab_bytes + (size_t)nprob * M.per + 256;
    return true;
}

template <class T>
static int fsm_many_run(const eik_grid *grid, const FsmManyPlan &MP, int nprob, const void *r,
                        const uint8_t *const *gamma, const void *const *g, void *const *u, int64_t max_sweeps,
                        void *ws, eik_fsm_stats *stats, cudaStream_t s) {
    const FsmPlan &P = MP.P;
    FsmMany<T> M;
    memset(&M, 0, sizeof(M));
    FsmArgs<T> &A = M.A;
    A.r = static_cast<const T *>(r);
    A.sy = grid->stride[1];
    A.nx = P.nx;
    A.ny = P.ny;
    A.nb = P.nb;
    A.nstepp = P.nstepp;
    A.h = (T)grid->h;
    A.max_sweeps = max_sweeps;
    // offsets of one problem's region (measured against a dummy base)
    char *const dummy = reinterpret_cast<char *>(256);
    FsmArgs<T> L;
    fsm_layout<T>(P, &L, dummy);
    M.o_state = reinterpret_cast<char *>(L.state) - dummy;
    M.o_rsk = reinterpret_cast<char *>(L.rsk) - dummy;
    M.o_ghands = reinterpret_cast<char *>(L.ghands) - dummy;
    M.o_gctl = reinterpret_cast<char *>(L.gctl) - dummy;
    M.o_dev = reinterpret_cast<char *>(L.dev) - dummy;
    M.tab = static_cast<const void *const *>(ws);
    M.ws0 = static_cast<char *>(ws) + MP.tab_bytes;
    M.per = MP.per;
    M.nprob = nprob;

    int rc, dev, optin = 0, nsm = 0;
    if ((rc = cuda_check(cudaGetDevice(&dev), "cudaGetDevice"))) return rc;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncAttributes fa;
    if ((rc = cuda_check(cudaFuncGetAttributes(&fa, k_fsmm_run<T>), "func attr"))) return rc;
    const bool single = (int)P.smem <= optin && P.nb <= 32 && regs_fit(fa, P.nb);
    // One warp a problem.  In FP64 only while the SMs have few of them: a warp that
    // has the FP64 pipe to itself is slow, but several share it, where the engine's
    // warps keep it full.  ms, one warp / engine: 32^2 (one column a lane) 152
    // problems 1.23 / 1.41, 304 1.67 / 1.86, 456 2.69 / 2.39, 1200 6.04 / 4.79; 33^2
    // (two) 152 1.88 / 1.98, 200 2.86 / 2.12, 456 5.05 / 3.02, 1200 12.2 / 6.65.
    int box_k = box2_use<T>(P.nx, P.ny);
    if (sizeof(T) == 8 && nprob > (box_k == 1 ? 2 : 1) * nsm) box_k = 0;
    // (a problem reads all of its own before it writes u, but others read then too)
    if (box_k && nprob > 1) {
        std::vector<Span> spans = {grid_span(r, grid, sizeof(T), nprob, false)};
        for (int p = 0; p < nprob; ++p) {
            spans.push_back(grid_span(gamma[p], grid, 1, p, false));
            spans.push_back(grid_span(g[p], grid, sizeof(T), p, false));
            spans.push_back(grid_span(u[p], grid, sizeof(T), p, true));
        }
        if (outputs_meet_inputs(spans)) box_k = 0;
    }
    const size_t box_smem = box2_smem_bytes<T>(P.nx, P.ny);
    const int nblk = (P.nb + P.wpc - 1) / P.wpc;
    int group = nprob;  // problems per cooperative launch
    if (box_k) {
        if ((rc = cuda_check(set_dyn_smem(fsmm_box_kernel<T>(box_k), (int)box_smem), "smem attr")))
            return rc;
    } else if (!single) {
        if ((rc = cuda_check(set_dyn_smem(k_fsmm_run_global<T>, (int)P.gsmem), "smem attr")))
            return rc;
        int per_sm = 0;
        if ((rc = cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fsmm_run_global<T>, 32 * P.wpc,
                                                                          P.gsmem), "occupancy")))
            return rc;
        group = std::min(nprob, per_sm * nsm / nblk);
        if (group < 1) {
            set_error("grid of %d x %d nodes needs %d co-resident CTAs, the device holds %d", P.nx, P.ny, nblk,
                      per_sm * nsm);
            return EIK_EUNSUPPORTED;
        }
    } else if ((rc = cuda_check(set_dyn_smem(k_fsmm_run<T>, (int)P.smem), "smem attr"))) {
        return rc;
    }
    // pointer table: gamma, g, u
    std::vector<const void *> tab((size_t)3 * nprob);
    for (int p = 0; p < nprob; ++p) {
        tab[p] = gamma[p];
        tab[nprob + p] = g[p];
        tab[2 * nprob + p] = u[p];
    }
    int nl = upload_ptrs(const_cast<const void **>(M.tab), tab.data(), 3 * nprob, s);
    if (nl < 0) return nl;
    if (box_k) {
        A.launches = nl + 1;
        EIK_LAUNCH("fsm_sweeps", s, fsmm_box_kernel<T>(box_k)<<<nprob, FSM_BOX_THREADS, box_smem, s>>>(M, stats));
        return cuda_check(cudaGetLastError(), "fsm launch");
    }
    const int ngroups = (nprob + group - 1) / group;
    nl += 2 + (single ? 1 : 1 + ngroups);
    A.launches = nl;
    A.multi = single ? 0 : 1;
    const size_t total = (size_t)P.nx * P.ny;
    const dim3 eg((unsigned)std::max<size_t>(1, std::min<size_t>((total + 255) / 256, (size_t)nsm * 16 / nprob + 1)),
                  (unsigned)nprob);
    EIK_LAUNCH("fsm_pack", s, k_fsmm_pack<T><<<eg, 256, 0, s>>>(M));
    if (single) {
        EIK_LAUNCH("fsm_sweeps", s, k_fsmm_run<T><<<nprob, 32 * P.nb, P.smem, s>>>(M));
    } else {
        EIK_LAUNCH("fsm_init", s, k_fsmm_init_global<T><<<nprob, 256, 0, s>>>(M));
        for (int p0 = 0; p0 < nprob; p0 += group) {
            int np = std::min(group, nprob - p0);
            void *args[] = {&M, &p0, const_cast<int *>(&nblk)};
            int tok = prof_begin("fsm_sweeps", s);
            rc = cuda_check(cudaLaunchCooperativeKernel((void *)k_fsmm_run_global<T>, np * nblk, 32 * P.wpc, args,
                                                        P.gsmem, s),
                            "fsm cooperative launch");
            prof_end(tok, s);
            if (rc) return rc;
        }
    }
    EIK_LAUNCH("fsm_unpack", s, k_fsmm_unpack<T><<<eg, 256, 0, s>>>(M, stats));
    return cuda_check(cudaGetLastError(), "fsm launch");
}
}  // namespace eik

using namespace eik;

extern "C" const char *eik_last_error(void) { return g_err; }

extern "C" int eik_version(void) { return 102; }

namespace eik {
int set_spin_limit_dd(long long);
int set_spin_limit_batch(long long);
int set_spin_limit_dd3(long long);
int set_spin_limit_fsm3(long long);
int set_spin_limit_adj(long long);
int set_spin_limit_dd1(long long);
}  // namespace eik

extern "C" int eik_set_wait_limit(int64_t iterations) {
    if (iterations < 0) {
        set_error("eik_set_wait_limit: iterations must be >= 0 (0 restores the default)");
        return EIK_EINVAL;
    }
    const long long v = iterations == 0 ? SPIN_LIMIT_DEFAULT : (long long)iterations;
    int (*const setters[])(long long) = {set_spin_limit_fsm, set_spin_limit_dd, set_spin_limit_batch,
                                         set_spin_limit_dd3, set_spin_limit_fsm3, set_spin_limit_adj,
                                         set_spin_limit_dd1};
    for (auto f : setters) {
        const int rc = cuda_check((cudaError_t)f(v), "cudaMemcpyToSymbol(wait limit)");
        if (rc) return rc;
    }
    return EIK_OK;
}

extern "C" int eik_profile_enable(int on) {
    int prev = g_prof_on ? 1 : 0;
    g_prof_on = on != 0;
    return prev;
}

extern "C" int eik_profile_collect(eik_kernel_time *out, int max_entries) {
    std::vector<eik_kernel_time> acc;
    int rc = EIK_OK;
    for (auto &r : g_prof) {
        float ms = 0.f;
        if (cudaEventSynchronize(r.b) != cudaSuccess || cudaEventElapsedTime(&ms, r.a, r.b) != cudaSuccess) {
            set_error("eik_profile_collect: event query failed");
            rc = EIK_ECUDA;
        }
        size_t k = 0;
        while (k < acc.size() && std::string(acc[k].name) != r.name) ++k;
        if (k == acc.size()) acc.push_back(eik_kernel_time{r.name, 0, 0.0, 0.0});
        acc[k].launches += 1;
        acc[k].total_ms += ms;
        if (ms > acc[k].max_ms) acc[k].max_ms = ms;
        g_prof_pool.push_back(r.a);
        g_prof_pool.push_back(r.b);
    }
    g_prof.clear();
    if (rc != EIK_OK) return rc;
    for (size_t k = 0; k < acc.size() && (int)k < max_entries; ++k) out[k] = acc[k];
    return (int)acc.size();
}

namespace eik {
// 3-D form (eik_fsm3.cu)
size_t fsm3_workspace_size(const eik_grid *grid, bool least);
int fsm3_run(const eik_grid *grid, const void *r, const uint8_t *gamma, const void *g, void *u, int64_t max_sweeps,
             void *ws, size_t ws_bytes, eik_fsm_stats *stats, cudaStream_t s);
}  // namespace eik

extern "C" size_t eik_fsm_workspace_size(const eik_grid *grid) {
    if (grid && grid->ndim == 3) return valid_grid_common(grid, 3) ? fsm3_workspace_size(grid, false) : 0;
    FsmPlan P;
    if (!fsm_plan(grid, P)) return 0;
    return P.bytes;
}

extern "C" int eik_fsm(const eik_grid *grid, const void *r, const uint8_t *gamma, const void *g, void *u,
                       int64_t max_sweeps, void *ws, size_t ws_bytes, eik_fsm_stats *stats, void *stream) {
    if (grid && grid->ndim == 3) {
        if (!valid_grid_common(grid, 3)) return EIK_EINVAL;
        if (!r || !gamma || !g || !u || !ws) {
            set_error("eik_fsm: NULL array argument");
            return EIK_EINVAL;
        }
        if (max_sweeps < 1 || max_sweeps > MAX_SWEEPS) {
            set_error("max_sweeps must be in [1, %lld]", MAX_SWEEPS);
            return EIK_EINVAL;
        }
        if (reinterpret_cast<uintptr_t>(ws) & 255) {
            set_error("workspace must be 256-byte aligned");
            return EIK_EINVAL;
        }
        const size_t need = fsm3_workspace_size(grid, true);
        if (ws_bytes < need) {
            set_error("workspace of %zu bytes is smaller than the %zu required", ws_bytes, need);
            return EIK_ENOMEM;
        }
        return fsm3_run(grid, r, gamma, g, u, max_sweeps, ws, ws_bytes, stats, static_cast<cudaStream_t>(stream));
    }
    FsmPlan P;
    if (!fsm_plan(grid, P)) return EIK_EINVAL;
    if (!r || !gamma || !g || !u || !ws) {
        set_error("eik_fsm: NULL array argument");
        return EIK_EINVAL;
    }
    if (max_sweeps < 1 || max_sweeps > MAX_SWEEPS || grid->n[1] > MAX_BOX_ROWS) {
        set_error("max_sweeps must be in [1, %lld] and n[1] <= %d", MAX_SWEEPS, MAX_BOX_ROWS);
        return EIK_EINVAL;
    }
    if (reinterpret_cast<uintptr_t>(ws) & 255) {
        set_error("workspace must be 256-byte aligned");
        return EIK_EINVAL;
    }
    if (ws_bytes < P.bytes) {
        set_error("workspace of %zu bytes is smaller than the %zu required", ws_bytes, P.bytes);
        return EIK_ENOMEM;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (grid->dtype == EIK_F64) return fsm_run<double>(grid, P, r, gamma, g, u, max_sweeps, ws, stats, s);
    return fsm_run<float>(grid, P, r, gamma, g, u, max_sweeps, ws, stats, s);
}

extern "C" size_t eik_fsm_many_workspace_size(const eik_grid *grid, int nprob) {
    FsmManyPlan M;
    if (!fsm_many_plan(grid, nprob, M)) return 0;
    return M.bytes;
}

extern "C" int eik_fsm_many(const eik_grid *grid, int nprob, const void *r, const uint8_t *const *gamma,
                            const void *const *g, void *const *u, int64_t max_sweeps, void *ws, size_t ws_bytes,
                            eik_fsm_stats *stats, void *stream) {
    FsmManyPlan M;
    if (!fsm_many_plan(grid, nprob, M)) return EIK_EINVAL;
    if (!r || !gamma || !g || !u || !ws) {
        set_error("eik_fsm_many: NULL argument");
        return EIK_EINVAL;
    }
    for (int p = 0; p < nprob; ++p) {
        if (!gamma[p] || !g[p] || !u[p]) {
            set_error("eik_fsm_many: NULL array of problem %d", p);
            return EIK_EINVAL;
        }
    }
    if (max_sweeps < 1 || max_sweeps > MAX_SWEEPS || grid->n[1] > MAX_BOX_ROWS) {
        set_error("max_sweeps must be in [1, %lld] and n[1] <= %d", MAX_SWEEPS, MAX_BOX_ROWS);
        return EIK_EINVAL;
    }
    if (reinterpret_cast<uintptr_t>(ws) & 255) {
        set_error("workspace must be 256-byte aligned");
        return EIK_EINVAL;
    }
    if (ws_bytes < M.bytes) {
        set_error("workspace of %zu bytes is smaller than the %zu required", ws_bytes, M.bytes);
        return EIK_ENOMEM;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (grid->dtype == EIK_F64) return fsm_many_run<double>(grid, M, nprob, r, gamma, g, u, max_sweeps, ws, stats, s);
    return fsm_many_run<float>(grid, M, nprob, r, gamma, g, u, max_sweeps, ws, stats, s);
}
