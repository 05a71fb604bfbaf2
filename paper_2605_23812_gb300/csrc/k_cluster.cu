// k_cluster.cu -- the pressure solve of one member in one thread-block cluster.
//
// The tiled kernels of k_poisson.cu run a V-cycle as six launches that re-read every vector from L2
// with halos, and its small levels leave all but one SM idle.  Here the blocks of a cluster hold a
// member's inner vectors on chip for the whole solve: residual, V-cycles, CG updates and the
// convergence tests of every refinement run in one launch, with no traffic but b, x and e.
//
// Layout.  The grid of the first level is cut into B x B blocks of cells (B = 4 or 2), one thread
// per block that holds fluid; solid blocks get no thread.  A thread keeps its block's iterate and
// right-hand side in registers, and the next log2(B) levels are local to it: restriction and
// prolongation are register sums.  Consecutive block rows form a slab per thread block of the
// cluster.  East / west neighbours come by shuffle, the others from a shared-memory plane that
// holds every thread's border cells; slab borders are pushed into the neighbouring block's plane
// with st.async, whose bytes complete a barrier there: 690 cycles from store to use, 465 to 665 for a
// barrier of the whole cluster (each measured by itself), but only the threads of a border wait for it.  The
// coarser levels are gathered in the cluster's first block and run the same way on its first warps
// (stages 1, 2), with a named barrier between half-sweeps.
//
// Red-black Gauss-Seidel does not depend on how cells are spread over threads, and every update
// uses the operations of the tiled kernels in their order, so FP32 iterates equal theirs bit for bit;
// dot products are df64 (or FP64) sums in another order, so a step length may round differently: runs of a
// few steps had the same bits in every case compared, runs of 30 000 steps differ in the eighth digit of J.
//
// Every wait on a barrier in shared memory has an iteration limit.  A thread whose wait ran out sends
// nothing more to other blocks and waits for nothing more, so the others' waits run out too; all blocks
// learn of it at the cluster barrier that ends a refinement (agree), leave together and mark the member's
// status as a solve that did not converge.
#include <algorithm>
#include <cstring>
#include <map>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/envar.h"
#include "df64.cuh"
#include "envar_internal.cuh"

namespace envar {

// ------------------------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ unsigned int sptr(const void *p) { return (unsigned int)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned int remote(unsigned int a, int rank)
{
    unsigned int r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void mb_init(unsigned int bar, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_expect(unsigned int bar, int bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mb_arrive_remote(unsigned int bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mb_try(unsigned int bar, unsigned int phase)
{
    unsigned int ok;
    asm volatile("{\n .reg .pred p;\n"
                 " mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(bar), "r"(phase)
                 : "memory");
    return ok != 0;
}
// a block's record of its waits
struct ClWatch {
    int failed;                      // one ran out
    int limit;                       // tries of a wait
    int any[2];                      // one ran out in some block of the cluster (agree; used in turn)
};
// per-thread flags
enum { CF_WLANE = 1, CF_ELANE = 2, CF_PUSH_S = 4, CF_PUSH_N = 8, CF_WAIT_S = 16, CF_WAIT_N = 32, CF_ACT = 64, CF_PAR = 128,
       CF_LOST = 256 };              // a wait of this thread ran out
// bounded wait; once one ran out, the block's other waits return at once.  A thread whose wait ran out
// neither sends to other blocks nor waits again.  (All of it behind the first try, which nearly always holds.)
__device__ __forceinline__ void mb_wait(unsigned int bar, unsigned int phase, ClWatch *w, int &flags)
{
    if (mb_try(bar, phase)) return;
    volatile ClWatch *v = w;
#pragma unroll 1
    for (int k = v->limit; k > 0 && !v->failed; --k)
        if (mb_try(bar, phase)) return;
    v->failed = 1;
    flags = (flags & ~(CF_PUSH_S | CF_PUSH_N | CF_WAIT_S | CF_WAIT_N)) | CF_LOST;
}
__device__ __forceinline__ bool has_failed(const ClWatch *w) { return *(const volatile int *)&w->failed != 0; }
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ int cluster_rank()
{
    int r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// asynchronous store into another block's shared memory, completing its bytes on that block's barrier
__device__ __forceinline__ void st_async(unsigned int a, float v, unsigned int bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(a), "f"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async(unsigned int a, double v, unsigned int bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(a), "d"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async2(unsigned int a, float v, float w, unsigned int bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(a), "f"(v), "f"(w), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async2(unsigned int a, double v, double w, unsigned int bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(a), "d"(v), "d"(w), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async4(unsigned int a, float v, float w, float x, float y, unsigned int bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a), "f"(v), "f"(w), "f"(x), "f"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ float ld_remote(unsigned int a, float)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ double ld_remote(unsigned int a, double)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

// ------------------------------------------------------------------------------------ plan (device view)
constexpr int CL_MAXC = 16;          // blocks per cluster at most
constexpr int CL_STAGES = 4;         // the cluster's levels, then up to three gathered stages
constexpr int CL_PAD = 4;            // columns left of a plane's cells (alignment of vector accesses)

struct ClSlab { int cb0, rb0, wb, hb, rxS, rxN; };   // block columns / rows held, blocks pushed in from south / north
struct ClStageArgs {
    int B, nlev, l0;                 // block size, levels, first level
    int bw, bh, nt;                  // blocks, threads (stage 0: per thread block)
    unsigned int rbw;                // 2^32 / bw rounded up
    int plane[3];                    // byte offset of each level's border plane in shared memory
    int pitch[3];                    // its row length (gathered stages; stage 0: from the slab's width)
    int rp;                          // byte offset of the residual plane handed to the next stage [bh][bw]
    int seq[3];                      // restriction from the level sums its four children in a row (else row pairs)
    // x-face, y-face conductances and smoothing factors of the threads' blocks, [value][record], copied to
    // shared memory (FP64, stage 0: left in global memory, for a second block per SM).  Stage 0: blocks with
    // equal values share a record (a cavity has a few dozen), so the tables fit: the V-cycle of 14 members at
    // 1024 x 512 took 53 us with the tables in L1, 45 us with them in shared memory.  Gathered stages: an
    // image per thread.
    const void *img[3];
    const int *kind[3];              // stage 0: each thread's record
    int nrec[3];
    int simg[3], sfm;                // gathered stages: byte offsets of their copies in shared memory
    int wide, ni, fo;                // a coarsest level of more cells than threads; cells in img; byte offset of f
    const int *fm;                   // per thread: fluid bits of its cells (16 | 4 << 16 | 1 << 20)
};
struct ClusterArgs {
    int C, nt, la, nst;
    int nu[2][2];                    // sweep pairs: [first level of the grid, others][pre, post]
    int coarse_sweeps;
    ClSlab slab[CL_MAXC];
    ClStageArgs st[CL_STAGES];
    const int4 *rec;                 // [C * nt] block (column | row << 16), flags | fluid bits << 16, open-face bits
    int nact;                        // blocks that hold fluid (gathered residuals)
    int sm_p, sm_lut, sm_red, sm_slot, sm_xs;   // byte offsets in shared memory
    int sm_idle;                     // zeros: the plane of threads without a block
    int sm_st;                       // copy of st for the gathered stages (indexed by a loop counter there; as kernel parameters: 2 to 4 % of a solve)
    int P;                           // pitch and member stride of the first level's arrays
    long long S;
};
struct SolveArgs {                   // one pressure solve (mode 0) or one V-cycle of the levels from la (mode 1)
    int mode, max_outer, first_o, one, count_last, max_inner, inner_guard;   // one: a single refinement (from first_o)
    int wait_limit;                  // tries of a wait in the kernel
    double inner_rtol2, rtol_abs;
    MixConst mc;
    double cxd, cyd;
    float cxf, cyf;
    int nx, ny;
    const uint8_t *fluid;
    const float *bh, *bl;
    float *xh, *xl;
    const double *b;
    double *x;
    void *acc;                       // the inner correction e
    const void *f;                   // mode 1: right-hand side and result of level la
    void *e;
    RedCtx rc;
    MemberCtl *ctl;
};

template <class T, int b> struct Blk { T v[b][b]; };

// shared memory of the kernel by byte offset (the compiler sees the address space)
template <class T> __device__ __forceinline__ T *sp(int off)
{
    extern __shared__ __align__(16) unsigned char sm[];
    return reinterpret_cast<T *>(sm + off);
}
__device__ __forceinline__ unsigned int sa32(int off) { return sptr(sp<unsigned char>(off)); }

// per-thread context of a stage
template <class T, int S> struct Ctx {
    int own[3];                      // byte offset of the block's first cell in each level's border plane
    int pitch[3];                    // its row length in bytes
    int flags, fm, kind[3];
    int tid, rank, id, nt;           // id: the stage
    // stage 0: remote rows for the pushes, halo barriers, exchange / gather / reduction counters
    unsigned int pushS[3], pushN[3], rbarS, rbarN;
    int rxS, rxN;
    int n, gat, nred;
    ClWatch *watch;
};
// barriers (byte offsets): halo south [2], halo north [2], reductions [2], gather, gathered result
enum { BAR_S = 0, BAR_N = 16, BAR_RED = 32, BAR_GAT = 48, BAR_RES = 56 };

// KIND 0: the cluster's blocks, 1: a gathered stage (named barrier id on its nt threads)
template <int KIND> __device__ __forceinline__ void stage_sync(int id, int nt)
{
    if constexpr (KIND == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nt) : "memory");
}

template <class T> __device__ __forceinline__ void ld_row(const T *p, T (&v)[4])
{
    if constexpr (sizeof(T) == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        const double2 q = *reinterpret_cast<const double2 *>(p), s = *reinterpret_cast<const double2 *>(p + 2);
        v[0] = q.x; v[1] = q.y; v[2] = s.x; v[3] = s.y;
    }
}
template <class T> struct V2;
template <> struct V2<float> { using type = float2; };
template <> struct V2<double> { using type = double2; };
template <class T> __device__ __forceinline__ void ld_row(const T *p, T (&v)[2])
{
    const typename V2<T>::type q = *reinterpret_cast<const typename V2<T>::type *>(p);
    v[0] = q.x; v[1] = q.y;
}
template <class T> __device__ __forceinline__ void ld_row(const T *p, T (&v)[1]) { v[0] = *p; }
template <class T> __device__ __forceinline__ void st_row(T *p, const T (&v)[4])
{
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2 *>(p + 2) = make_double2(v[2], v[3]);
    }
}
template <class T> __device__ __forceinline__ void st_row(T *p, const T (&v)[2])
{
    *reinterpret_cast<typename V2<T>::type *>(p) = typename V2<T>::type{v[0], v[1]};
}
template <class T> __device__ __forceinline__ void st_row(T *p, const T (&v)[1]) { *p = v[0]; }
template <class T, int b> __device__ __forceinline__ void push_row(unsigned int a, const T (&v)[b], unsigned int bar)
{
    // as few stores as possible: each lane's store completes its bytes on the barrier by itself
    if constexpr (b == 1) {
        st_async(a, v[0], bar);
    } else if constexpr (b == 4 && sizeof(T) == 4) {
        st_async4(a, v[0], v[1], v[2], v[3], bar);
    } else {
#pragma unroll
        for (int i = 0; i < b; i += 2) st_async2(a + i * (int)sizeof(T), v[i], v[i + 1], bar);
    }
}
// global rows of a block (L2: other thread blocks of the cluster write them)
__device__ __forceinline__ void ldg_row(const float *p, float (&v)[4]) { const float4 q = __ldcg(reinterpret_cast<const float4 *>(p)); v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w; }
__device__ __forceinline__ void ldg_row(const float *p, float (&v)[2]) { const float2 q = __ldcg(reinterpret_cast<const float2 *>(p)); v[0] = q.x; v[1] = q.y; }
__device__ __forceinline__ void ldg_row(const double *p, double (&v)[2]) { const double2 q = __ldcg(reinterpret_cast<const double2 *>(p)); v[0] = q.x; v[1] = q.y; }
__device__ __forceinline__ void ldg_row(const double *p, double (&v)[4])
{
    const double2 q = __ldcg(reinterpret_cast<const double2 *>(p)), s = __ldcg(reinterpret_cast<const double2 *>(p + 2));
    v[0] = q.x; v[1] = q.y; v[2] = s.x; v[3] = s.y;
}

// ------------------------------------------------------------------------------------ border exchange
// Make the border cells of every block visible to its neighbours: into the stage's plane, and (stage
// 0) into the neighbouring slabs' planes.  Two halo barriers per side, used in turn: a neighbour can
// be at most one exchange ahead (its next push waits for this block's), so its bytes never meet the
// barrier of the exchange before.
//
// A halo row has one buffer, and a neighbour may push the next one while this block still reads it: it waited
// for this block's push of the same exchange, which comes before the read.  The same holds for a block's own
// border cells in its plane, which it stores without waiting for the last read of them.  Both rely on this, and
// every use has to keep it:
//   - two exchanges of a plane with nothing between them but a half-sweep differ only in the colour that the
//     half-sweep updates, and it reads the other one: what it reads is overwritten with the same values;
//   - a read of both colours (residual, q = A p) is followed by an exchange of another level's plane, by the
//     gather or by a sum over the cluster before the plane is written again, and none of these gets
//     past a block that has not finished the read.
template <class T, int b, int S, bool MULTI>
__device__ __forceinline__ void exchange(Ctx<T, S> &c, int k, const T (&e)[b][b])
{
    // (threads without a block keep zeros in a plane of their own: no branch)
    const int o = c.own[k], p = c.pitch[k];
    bool dead = false;
    if constexpr (S == 0 && MULTI) dead = has_failed(c.watch);
    if constexpr (S == 0 && MULTI) {
        const unsigned int off = 8u * (c.n & 1);
        if (c.flags & (CF_PUSH_S | CF_PUSH_N)) {
            if (c.flags & CF_PUSH_S) push_row<T, b>(c.pushS[k], e[0], c.rbarS + off);
            if (c.flags & CF_PUSH_N) push_row<T, b>(c.pushN[k], e[b - 1], c.rbarN + off);
        }
    }
    st_row(sp<T>(o), e[0]);
    if constexpr (b > 1) st_row(sp<T>(o + (b - 1) * p), e[b - 1]);
    if constexpr (b > 2) {
        if ((c.flags & (CF_WLANE | CF_ELANE)) != (CF_WLANE | CF_ELANE)) {
#pragma unroll
            for (int r = 1; r < b - 1; ++r) st_row(sp<T>(o + r * p), e[r]);
        }
    }
    if constexpr (S == 0 && MULTI) {
        const unsigned int off = 8u * (c.n & 1), ph = (c.n >> 1) & 1;
        // (a barrier whose bytes did not come is not armed a second time: the block's waits of the exchange
        // before last, which used this one, ended ahead of the last exchange's __syncthreads)
        if (c.tid == 0 && !dead) {
            if (c.rxS) mb_expect(sa32(BAR_S) + off, c.rxS * b * (int)sizeof(T));
            if (c.rxN) mb_expect(sa32(BAR_N) + off, c.rxN * b * (int)sizeof(T));
        }
        __syncthreads();
        if (c.flags & (CF_WAIT_S | CF_WAIT_N)) {
            if (c.flags & CF_WAIT_S) mb_wait(sa32(BAR_S) + off, ph, c.watch, c.flags);
            if (c.flags & CF_WAIT_N) mb_wait(sa32(BAR_N) + off, ph, c.watch, c.flags);
        }
        c.n++;
        __syncwarp();
    } else {
        stage_sync<S>(c.id, c.nt);
    }
}

// Neighbours outside the block: rows below / above from the plane; columns from the plane too (blocks
// of at most 2 x 2 cells, which the plane holds whole), or by shuffle where the neighbour is the
// adjacent lane.
template <class T, int b, int S>
__device__ __forceinline__ void rows_sn(const Ctx<T, S> &c, int k, T (&s)[b], T (&n)[b])
{
    ld_row(sp<const T>(c.own[k] - c.pitch[k]), s);
    ld_row(sp<const T>(c.own[k] + b * c.pitch[k]), n);
}
template <class T, int b, int S> __device__ __forceinline__ T west(const Ctx<T, S> &c, int k, const T (&e)[b][b], int r)
{
    const T *pl = sp<const T>(c.own[k] + r * c.pitch[k]);
    if constexpr (b <= 2) return pl[-1];
    else {
        T w = __shfl_up_sync(0xffffffffu, e[r][b - 1], 1);
        if (!(c.flags & CF_WLANE)) w = pl[-1];
        return w;
    }
}
template <class T, int b, int S> __device__ __forceinline__ T east(const Ctx<T, S> &c, int k, const T (&e)[b][b], int r)
{
    const T *pl = sp<const T>(c.own[k] + r * c.pitch[k]);
    if constexpr (b <= 2) return pl[b];
    else {
        T w = __shfl_down_sync(0xffffffffu, e[r][0], 1);
        if (!(c.flags & CF_ELANE)) w = pl[b];
        return w;
    }
}

// ------------------------------------------------------------------------------------ half-sweeps
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// Conductances (and smoothing factors 1 / sum) of a block of a level with explicit conductances: in
// registers for 2 x 2 and 1 x 1 blocks, read at each use for 4 x 4 blocks (56 values).
template <class T, int b> struct Cond {
    T x_[b][b + 1], y_[b + 1][b], v_[b][b];
    __device__ __forceinline__ T x(int r, int i) const { return x_[r][i]; }
    __device__ __forceinline__ T y(int r, int i) const { return y_[r][i]; }
    __device__ __forceinline__ T v(int r, int i) const { return v_[r][i]; }
    // img: [value][record], n records
    __device__ __forceinline__ void load(const T *img, int n)
    {
        const T *q = img;
#pragma unroll
        for (int r = 0; r < b; ++r)
#pragma unroll
            for (int i = 0; i <= b; ++i, q += n) x_[r][i] = *q;
#pragma unroll
        for (int r = 0; r <= b; ++r)
#pragma unroll
            for (int i = 0; i < b; ++i, q += n) y_[r][i] = *q;
#pragma unroll
        for (int r = 0; r < b; ++r)
#pragma unroll
            for (int i = 0; i < b; ++i, q += n) v_[r][i] = *q;
    }
};
template <class T> struct Cond<T, 4> {
    int o, n;                        // byte offset of the record
    __device__ __forceinline__ T x(int r, int i) const { return sp<const T>(o)[(r * 5 + i) * n]; }
    __device__ __forceinline__ T y(int r, int i) const { return sp<const T>(o)[(20 + r * 4 + i) * n]; }
    __device__ __forceinline__ T v(int r, int i) const { return sp<const T>(o)[(40 + r * 4 + i) * n]; }
    __device__ __forceinline__ void load(const T *img, int n_) { o = (int)(reinterpret_cast<const unsigned char *>(img) - sp<const unsigned char>(0)); n = n_; }
};

// uniform conductances and open-face bits (the grid's first level)
template <class T, int b> struct Open {
    T cx, cy;
    const T *lut;                    // [16] sum of the open faces' conductances, [16] its inverse
    unsigned int lo, hi;             // 4 open-face bits per cell, row by row
    bool all;                        // all of the warp's cells have four open faces
    __device__ __forceinline__ unsigned int bits(int r, int i) const
    {
        const int q = 4 * (r * b + i);
        return (q < 32 ? lo >> (q & 31) : hi >> (q & 31)) & 15u;
    }
};

// one half-sweep: the cells of one colour; zero: the iterate is zero, so the update is v f
template <class T, int b, int S>
__device__ __forceinline__ void half_sweep(const Ctx<T, S> &c, int k, int col, const Cond<T, b> &q, const T (&f)[b][b],
                                           T (&e)[b][b])
{
    T s[b], n[b];
    rows_sn<T, b, S>(c, k, s, n);
    if constexpr (b == 1) {
        const T w = west<T, b, S>(c, k, e, 0), o = east<T, b, S>(c, k, e, 0);
        T acc = fma_(q.x(0, 0), w, f[0][0]);
        acc = fma_(q.x(0, 1), o, acc);
        acc = fma_(q.y(0, 0), s[0], acc);
        acc = fma_(q.y(1, 0), n[0], acc);
        acc = q.v(0, 0) * acc;
        e[0][0] = ((c.flags & CF_PAR) != 0) == (col != 0) ? acc : e[0][0];
    } else {
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
            if (cc != col) continue;
            T sd[b];
#pragma unroll
            for (int r = 0; r < b; ++r) sd[r] = ((cc ^ r) & 1) == 0 ? west<T, b, S>(c, k, e, r) : east<T, b, S>(c, k, e, r);
#pragma unroll
            for (int r = 0; r < b; ++r) {
                const int p = (cc ^ r) & 1;
                const T side = sd[r];
#pragma unroll
                for (int i = 0; i < b; ++i) {
                    if ((i & 1) != p) continue;
                    const T w = i > 0 ? e[r][i > 0 ? i - 1 : 0] : side, o = i < b - 1 ? e[r][i < b - 1 ? i + 1 : 0] : side;
                    const T ss = r > 0 ? e[r > 0 ? r - 1 : 0][i] : s[i], nn = r < b - 1 ? e[r < b - 1 ? r + 1 : 0][i] : n[i];
                    T acc = fma_(q.x(r, i), w, f[r][i]);
                    acc = fma_(q.x(r, i + 1), o, acc);
                    acc = fma_(q.y(r, i), ss, acc);
                    acc = fma_(q.y(r + 1, i), nn, acc);
                    e[r][i] = q.v(r, i) * acc;
                }
            }
        }
    }
}
template <class T, int b, int S, bool ALL>
__device__ __forceinline__ void half_open(const Ctx<T, S> &c, int k, int col, const Open<T, b> &q, const T (&f)[b][b], T (&e)[b][b])
{
    T s[b], n[b];
    rows_sn<T, b, S>(c, k, s, n);
    const T vall = q.lut[31];
#pragma unroll
    for (int cc = 0; cc < 2; ++cc) {
        if (cc != col) continue;
        T sd[b];
#pragma unroll
        for (int r = 0; r < b; ++r) sd[r] = ((cc ^ r) & 1) == 0 ? west<T, b, S>(c, k, e, r) : east<T, b, S>(c, k, e, r);
#pragma unroll
        for (int r = 0; r < b; ++r) {
            const int p = (cc ^ r) & 1;
#pragma unroll
            for (int i = 0; i < b; ++i) {
                if ((i & 1) != p) continue;
                const T w = i > 0 ? e[r][i > 0 ? i - 1 : 0] : sd[r], o = i < b - 1 ? e[r][i < b - 1 ? i + 1 : 0] : sd[r];
                const T ss = r > 0 ? e[r > 0 ? r - 1 : 0][i] : s[i], nn = r < b - 1 ? e[r < b - 1 ? r + 1 : 0][i] : n[i];
                e[r][i] = (ALL ? vall : q.lut[16 + q.bits(r, i)]) * fma_(q.cy, ss + nn, fma_(q.cx, w + o, f[r][i]));
            }
        }
    }
}
// q.all: every cell of the warp has four open faces, one smoothing factor for all
template <class T, int b, int S>
__device__ __forceinline__ void half_sweep(const Ctx<T, S> &c, int k, int col, const Open<T, b> &q, const T (&f)[b][b],
                                           T (&e)[b][b])
{
    if (q.all) half_open<T, b, S, true>(c, k, col, q, f, e);
    else half_open<T, b, S, false>(c, k, col, q, f, e);
}
template <class T, int b, int S>
__device__ __forceinline__ void first_half(const Ctx<T, S> &c, const Cond<T, b> &q, const T (&f)[b][b], T (&e)[b][b])
{
#pragma unroll
    for (int r = 0; r < b; ++r)
#pragma unroll
        for (int i = 0; i < b; ++i)
            e[r][i] = (b == 1 ? !(c.flags & CF_PAR) : !((r ^ i) & 1)) ? q.v(r, i) * f[r][i] : (T)0;
}
template <class T, int b, int S>
__device__ __forceinline__ void first_half(const Ctx<T, S> &c, const Open<T, b> &q, const T (&f)[b][b], T (&e)[b][b])
{
#pragma unroll
    for (int r = 0; r < b; ++r)
#pragma unroll
        for (int i = 0; i < b; ++i) e[r][i] = !((r ^ i) & 1) ? q.lut[16 + q.bits(r, i)] * f[r][i] : (T)0;
}

// residual f - A e of cell (r, i) from its neighbours; seq: the coarse block's rounding (the diagonal
// term by itself), else the tiled smoothers' (the west term by itself)
template <class T, int b>
__device__ __forceinline__ T cell_res(const Cond<T, b> &q, int r, int i, T f, T e, T w, T o, T s, T n, int seq)
{
    const T kw = q.x(r, i), ke = q.x(r, i + 1), ks = q.y(r, i), kn = q.y(r + 1, i);
    const T d = ((kw + ke) + ks) + kn;
    T ax = seq ? fma_(-kw, w, d * e) : fma_(d, e, -(kw * w));
    ax = fma_(-ke, o, ax);
    ax = fma_(-ks, s, ax);
    ax = fma_(-kn, n, ax);
    return f - ax;
}
template <class T, int b>
__device__ __forceinline__ T cell_res(const Open<T, b> &q, int r, int i, T f, T e, T w, T o, T s, T n, int)
{
    const unsigned int t = q.bits(r, i);
    const T ax = fma_(-q.cy, s + n, fma_(q.lut[t], e, -(q.cx * (w + o))));
    return t ? f - ax : f;
}
template <class T, int b, int S, class Q>
__device__ __forceinline__ void residual(const Ctx<T, S> &c, int k, const Q &q, int seq, const T (&f)[b][b], const T (&e)[b][b], T (&res)[b][b])
{
    T s[b], n[b];
    rows_sn<T, b, S>(c, k, s, n);
#pragma unroll
    for (int r = 0; r < b; ++r) {
        const T wv = west<T, b, S>(c, k, e, r), ev = east<T, b, S>(c, k, e, r);
#pragma unroll
        for (int i = 0; i < b; ++i) {
            const T w = i > 0 ? e[r][i > 0 ? i - 1 : 0] : wv, o = i < b - 1 ? e[r][i < b - 1 ? i + 1 : 0] : ev;
            const T ss = r > 0 ? e[r > 0 ? r - 1 : 0][i] : s[i], nn = r < b - 1 ? e[r < b - 1 ? r + 1 : 0][i] : n[i];
            res[r][i] = cell_res<T, b>(q, r, i, f[r][i], e[r][i], w, o, ss, nn, seq);
        }
    }
}
// the four children of a coarse cell, summed as the tiled smoothers (row pairs) or the coarse block
// (one after the other) do
template <class T> __device__ __forceinline__ T sum4(T a, T b, T c, T d, int seq)
{
    return seq ? ((a + b) + c) + d : (a + b) + (c + d);
}

// ------------------------------------------------------------------------------------ V-cycle
// half-sweeps from .. 2 pairs - 1 from the present iterate, colours c0, c0 ^ 1, ...; each is followed by
// an exchange, but (skip_last) not the last one
template <class T, int b, int S, bool MULTI, class Q>
__device__ __forceinline__ void sweeps(Ctx<T, S> &c, int k, int from, int pairs, int c0, bool skip_last, const Q &q, const T (&f)[b][b],
                                       T (&e)[b][b])
{
    const int n = 2 * pairs - (skip_last ? 1 : 0);
    int s = from;
#pragma unroll 1
    for (; s < n; ++s) {
        half_sweep<T, b, S>(c, k, (s & 1) ^ c0, q, f, e);
        exchange<T, b, S, MULTI>(c, k, e);
    }
    if (skip_last) half_sweep<T, b, S>(c, k, (s & 1) ^ c0, q, f, e);
}

template <class T, int b, int S>
__device__ __forceinline__ void load_cond(const ClusterArgs &a, const Ctx<T, S> &c, int k, Cond<T, b> &q)
{
    const ClStageArgs &st = S > 0 ? sp<const ClStageArgs>(a.sm_st)[c.id] : a.st[0];
    if constexpr (S > 0) q.load(sp<const T>(st.simg[k]) + c.tid, st.nt);
    else if constexpr (sizeof(T) == 4) q.load(sp<const T>(st.simg[k]) + c.kind[k], st.nrec[k]);
    else q.load(reinterpret_cast<const T *>(st.img[k]) + c.kind[k], st.nrec[k]);
}

template <class T, int b, int S, bool MULTI, class Q>
__device__ __forceinline__ void descend(Ctx<T, S> &c, int k, int pre, const Q &q, const T (&f)[b][b], T (&e)[b][b])
{
    first_half<T, b, S>(c, q, f, e);
    exchange<T, b, S, MULTI>(c, k, e);
    sweeps<T, b, S, MULTI>(c, k, 1, pre, 0, false, q, f, e);
}
template <class T, int b, int S, bool MULTI, class Q>
__device__ __forceinline__ void ascend(Ctx<T, S> &c, int k, int post, const Q &q, const T (&f)[b][b], T (&e)[b][b])
{
    exchange<T, b, S, MULTI>(c, k, e);
    sweeps<T, b, S, MULTI>(c, k, 0, post, 1, true, q, f, e);
}
// coarse correction onto the fluid cells (bit r b + i of m)
template <class T, int b> __device__ __forceinline__ void prolong(unsigned int m, const T (&ec)[b / 2][b / 2], T (&e)[b][b])
{
#pragma unroll
    for (int r = 0; r < b; ++r)
#pragma unroll
        for (int i = 0; i < b; ++i)
            if (m >> (r * b + i) & 1u) e[r][i] += ec[r / 2][i / 2];
}

// The gathered stages on the first threads of the cluster's first block (or of the only one): the
// residual plane of the stage before is a stage's right-hand side, its plane of level 0 receives its
// result.  One copy of the code runs every stage (the instructions of a V-cycle have to stay in the
// instruction cache: with a copy per stage the whole kernel was 420 KB and ran at half the speed);
// each stage's iterates wait in local memory while the deeper ones run.
template <class T> __device__ __forceinline__ void gathered(const ClusterArgs &a, int tid)
{
    const ClStageArgs *sst = sp<const ClStageArgs>(a.sm_st);
    T save[CL_STAGES][10];
    Ctx<T, 1> c;
    c.tid = tid; c.rank = 0;
    T f[2][2], e[2][2], f1[1][1], e1[1][1];
    auto enter = [&](int s) {
        const ClStageArgs &st = sst[s];
        c.id = s; c.nt = st.nt;
        const bool act = tid < st.bw * st.bh;
        // tid / bw by the stage's reciprocal (exact for tid < 2^16)
        const int by = act ? (int)__umulhi((unsigned int)tid, st.rbw) : 0, bx = act ? tid - by * st.bw : 0;
        c.flags = (act ? CF_ACT : 0) | (((bx ^ by) & 1) ? CF_PAR : 0);
        c.fm = act ? sp<const int>(st.sfm)[tid] : 0;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            // level k of the stage, counted from its 2 x 2 level: a stage of single cells has only k = 1
            const int b = 2 >> k, kk = st.B == 2 ? k : 0;
            c.pitch[k] = act ? st.pitch[kk] * (int)sizeof(T) : 128;
            c.own[k] = act ? st.plane[kk] + (by * b + 1) * c.pitch[k] + (CL_PAD + bx * b) * (int)sizeof(T) : a.sm_idle + 128 + 32;
        }
        return int2{bx, by};
    };
    auto cond1 = [&](Cond<T, 1> &q) {
        const ClStageArgs &st = sst[c.id];
        q.load(sp<const T>(st.simg[st.B == 2 ? 1 : 0]) + tid, st.nt);
    };
    int s = 1;
    for (;; ++s) {                                           // down
        const ClStageArgs &st = sst[s], &up = sst[s - 1];
        const int2 xy = enter(s);
        const bool act = (c.flags & CF_ACT) != 0, last = s + 1 == a.nst;
        const int seq = up.seq[up.nlev - 1];
        const int rp = up.rp + (2 * st.B) * (xy.y * up.bw + xy.x) * (int)sizeof(T), rw = up.bw * (int)sizeof(T);
        if (st.B == 2) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                T lo[4], hi[4];                              // up.bw = 4 bw: aligned rows of four
                ld_row(sp<const T>(rp + 2 * r * rw), lo);
                ld_row(sp<const T>(rp + (2 * r + 1) * rw), hi);
                f[r][0] = act ? sum4(lo[0], lo[1], hi[0], hi[1], seq) : (T)0;
                f[r][1] = act ? sum4(lo[2], lo[3], hi[2], hi[3], seq) : (T)0;
            }
            Cond<T, 2> q;
            load_cond<T, 2, 1>(a, c, 0, q);
            descend<T, 2, 1, false>(c, 0, a.nu[1][0], q, f, e);
            T res[2][2];
            residual<T, 2, 1>(c, 0, q, st.seq[0], f, e, res);
            f1[0][0] = sum4(res[0][0], res[0][1], res[1][0], res[1][1], st.seq[0]);
        } else {
            T lo[2], hi[2];
            ld_row(sp<const T>(rp), lo);
            ld_row(sp<const T>(rp + rw), hi);
            f1[0][0] = act ? sum4(lo[0], lo[1], hi[0], hi[1], seq) : (T)0;
        }
        Cond<T, 1> q;
        cond1(q);
        descend<T, 1, 1, false>(c, 1, last ? a.coarse_sweeps : a.nu[1][0], q, f1, e1);
        if (last) break;
        T res[1][1];
        residual<T, 1, 1>(c, 1, q, st.seq[st.nlev - 1], f1, e1, res);
        if (act) *sp<T>(st.rp + (xy.y * st.bw + xy.x) * (int)sizeof(T)) = res[0][0];
        stage_sync<1>(s, st.nt);
        if (tid >= sst[s + 1].nt) break;
        T *sv = save[s];
        sv[0] = f[0][0]; sv[1] = f[0][1]; sv[2] = f[1][0]; sv[3] = f[1][1];
        sv[4] = e[0][0]; sv[5] = e[0][1]; sv[6] = e[1][0]; sv[7] = e[1][1];
        sv[8] = f1[0][0]; sv[9] = e1[0][0];
    }
    for (bool fresh = true; s >= 1; --s, fresh = false) {    // up
        const ClStageArgs &st = sst[s];
        const bool last = s + 1 == a.nst;
        if (!fresh) {
            const T *sv = save[s];
            f[0][0] = sv[0]; f[0][1] = sv[1]; f[1][0] = sv[2]; f[1][1] = sv[3];
            e[0][0] = sv[4]; e[0][1] = sv[5]; e[1][0] = sv[6]; e[1][1] = sv[7];
            f1[0][0] = sv[8]; e1[0][0] = sv[9];
        }
        const int2 xy = enter(s);
        const bool act = (c.flags & CF_ACT) != 0;
        if (!last) {
            stage_sync<1>(s, st.nt);                         // the deeper stages' result is complete
            const ClStageArgs &nx = sst[s + 1];
            const T ec = *sp<const T>(nx.plane[0] + (((xy.y >> 1) + 1) * nx.pitch[0] + CL_PAD + (xy.x >> 1)) * (int)sizeof(T));
            if (c.fm >> 20 & 1) e1[0][0] += ec;
        }
        Cond<T, 1> q;
        cond1(q);
        ascend<T, 1, 1, false>(c, 1, last ? a.coarse_sweeps : a.nu[1][1], q, f1, e1);
        if (st.B == 2) {
            prolong<T, 2>((unsigned int)(c.fm >> 16) & 15u, e1, e);
            Cond<T, 2> q2;
            load_cond<T, 2, 1>(a, c, 0, q2);
            ascend<T, 2, 1, false>(c, 0, a.nu[1][1], q2, f, e);
            if (act) {
                st_row(sp<T>(c.own[0]), e[0]);
                st_row(sp<T>(c.own[0] + c.pitch[0]), e[1]);
            }
        } else if (act) {
            *sp<T>(c.own[1]) = e1[0][0];
        }
    }
}

// A coarsest level of more cells than the block has threads (an odd level of a large grid: 672 x 400 ends
// at 42 x 25): iterate, right-hand side and conductances in shared memory, the cells of a colour dealt
// out to the threads.  Without it such a grid runs the levels from 1 on as eight launches per V-cycle.
template <class T> __device__ __forceinline__ void gathered_wide(const ClusterArgs &a, int tid)
{
    const ClStageArgs &st = a.st[1], &up = a.st[0];
    const int bw = st.bw, nt = st.nt, ni = st.ni, pitch = st.pitch[0], seq = up.seq[up.nlev - 1];
    T *f = sp<T>(st.fo), *e = sp<T>(st.plane[0]) + pitch + CL_PAD;
    const T *im = sp<const T>(st.simg[0]), *rp = sp<const T>(up.rp);
    for (int q = tid; q < bw * st.bh; q += nt) {
        const int y = (int)__umulhi((unsigned int)q, st.rbw), x = q - y * bw;
        const T *lo = rp + 2 * y * up.bw + 2 * x, *hi = lo + up.bw;
        f[q] = sum4(lo[0], lo[1], hi[0], hi[1], seq);
        e[y * pitch + x] = (T)0;
    }
    stage_sync<1>(1, nt);
    const int hw = (bw + 1) / 2;                             // at most one cell of a colour per pair of columns
    const unsigned int rhw = 0xffffffffu / (unsigned int)hw + 1u;
    auto half = [&](int col, bool zero) {
        for (int q = tid; q < hw * st.bh; q += nt) {
            const int y = (int)__umulhi((unsigned int)q, rhw), x = 2 * (q - y * hw) + ((y ^ col) & 1);
            if (x < bw) {
                const int at = y * bw + x;
                T *c = e + y * pitch + x;
                T acc = f[at];
                if (!zero) {
                    acc = fma_(im[at], c[-1], acc);
                    acc = fma_(im[ni + at], c[1], acc);
                    acc = fma_(im[2 * ni + at], c[-pitch], acc);
                    acc = fma_(im[3 * ni + at], c[pitch], acc);
                }
                *c = im[4 * ni + at] * acc;
            }
        }
        stage_sync<1>(1, nt);
    };
    for (int h = 0; h < 2 * a.coarse_sweeps; ++h) half(h & 1, h == 0);
    for (int h = 0; h < 2 * a.coarse_sweeps; ++h) half((h & 1) ^ 1, false);
}
template <class T> __device__ __forceinline__ void gathered_any(const ClusterArgs &a, int tid)
{
    if (sizeof(T) == 4 && a.st[1].wide) gathered_wide<T>(a, tid);
    else gathered<T>(a, tid);
}

// hand the residual of the cluster's last level to the gathered stages and return the coarse
// correction of this thread's cell
template <class T, bool MULTI> __device__ __forceinline__ T gather_stage(const ClusterArgs &a, Ctx<T, 0> &c, T res)
{
    const ClStageArgs &st = a.st[0], &nx = a.st[1];
    const int xy = a.rec[c.rank * st.nt + c.tid].x;
    const int bx = xy & 0xffff, by = (xy >> 16) & 0xffff;
    const int at = st.rp + (by * st.bw + bx) * (int)sizeof(T);
    const int from = nx.plane[0] + (((by >> 1) + 1) * nx.pitch[0] + CL_PAD + (bx >> 1)) * (int)sizeof(T);
    const bool act = (c.flags & CF_ACT) != 0;
    if constexpr (MULTI) {
        const unsigned int gbar = sa32(BAR_GAT), rbar = sa32(BAR_RES);
        const unsigned int ph = c.gat & 1;
        // (threads whose own waits were met send one gather more at most, as they wait for its result)
        if (!(c.flags & CF_LOST)) {
            if (c.rank == 0 && c.tid == 0) mb_expect(gbar, a.nact * (int)sizeof(T));
            if (act) st_async(remote(sa32(at), 0), res, remote(gbar, 0));
        }
        if (c.rank == 0 && c.tid < nx.nt) {
            if (!(c.flags & CF_LOST)) mb_wait(gbar, ph, c.watch, c.flags);
            __syncwarp();
            gathered_any<T>(a, c.tid);
            stage_sync<1>(1, nx.nt);
            if (c.tid < a.C && !(c.flags & CF_LOST)) {
                asm volatile("fence.acq_rel.cluster;" ::: "memory");
                mb_arrive_remote(remote(rbar, c.tid));
            }
            __syncwarp();
        }
        if (!(c.flags & CF_LOST)) mb_wait(rbar, ph, c.watch, c.flags);
        c.gat++;
        __syncwarp();
        return act ? ld_remote(remote(sa32(from), 0), (T)0) : (T)0;
    } else {
        if (act) *sp<T>(at) = res;
        __syncthreads();
        if (c.tid < nx.nt) gathered_any<T>(a, c.tid);
        __syncthreads();
        return act ? *sp<const T>(from) : (T)0;
    }
}

// level k of the cluster's levels (b x b cells per thread): f -> e, one symmetric V-cycle from here down
template <class T, int b, bool MULTI>
__device__ __forceinline__ void vlevel(const ClusterArgs &a, Ctx<T, 0> &c, int k, const T (&f)[b][b], T (&e)[b][b])
{
    const ClStageArgs &st = a.st[0];
    const int first = st.l0 + k == 0 ? 0 : 1;
    Cond<T, b> q;
    load_cond<T, b, 0>(a, c, k, q);
    descend<T, b, 0, MULTI>(c, k, a.nu[first][0], q, f, e);
    T res[b][b];
    residual<T, b, 0>(c, k, q, st.seq[k], f, e, res);
    if constexpr (b > 1) {
        T fc[b / 2][b / 2], ec[b / 2][b / 2];
#pragma unroll
        for (int r = 0; r < b / 2; ++r)
#pragma unroll
            for (int i = 0; i < b / 2; ++i)
                fc[r][i] = sum4(res[2 * r][2 * i], res[2 * r][2 * i + 1], res[2 * r + 1][2 * i], res[2 * r + 1][2 * i + 1], st.seq[k]);
        vlevel<T, b / 2, MULTI>(a, c, k + 1, fc, ec);
        prolong<T, b>((unsigned int)(b == 4 ? c.fm & 0xffff : (c.fm >> 16) & 15), ec, e);
    } else {
        const T ec = gather_stage<T, MULTI>(a, c, res[0][0]);
        if (c.fm >> 20 & 1) e[0][0] += ec;
    }
    load_cond<T, b, 0>(a, c, k, q);
    ascend<T, b, 0, MULTI>(c, k, a.nu[first][1], q, f, e);
}

// ------------------------------------------------------------------------------------ reductions
__device__ __forceinline__ f2 wsum(f2 v) { return warp_sum_df(v); }
__device__ __forceinline__ double wsum(double v) { return warp_sum(v); }
__device__ __forceinline__ f2 as_acc(double d, f2) { return f2{__int_as_float(__double2loint(d)), __int_as_float(__double2hiint(d))}; }
__device__ __forceinline__ double as_acc(double d, double) { return d; }
__device__ __forceinline__ double as_bits(f2 v) { return __hiloint2double(__float_as_int(v.l), __float_as_int(v.h)); }
__device__ __forceinline__ double as_bits(double v) { return v; }

// Sum (or, is_max, maximum) over the cluster's threads in a fixed order; warp 0's lanes hold the total.
// The caller synchronises before the next use.  Slots by rank, two sets used in turn.
template <class T, class V, bool MULTI, bool MAX>
__device__ __forceinline__ V cluster_total(const ClusterArgs &a, Ctx<T, 0> &c, V v)
{
    double *red = sp<double>(a.sm_red);
    const int lane = c.tid & 31, w = c.tid >> 5, nw = (a.nt + 31) >> 5;
    auto comb = [](V x) {
        if constexpr (MAX) return warp_max(x);
        else return wsum(x);
    };
    v = comb(v);
    if (lane == 0) red[w] = as_bits(v);
    __syncthreads();
    V tot{};
    if (w == 0) {
        V x{};
        if (lane < nw) x = as_acc(red[lane], V{});
        tot = comb(x);
        if constexpr (MULTI) {
            const int par = c.nred & 1;
            const unsigned int bar = sa32(BAR_RED) + 8u * par;
            const unsigned int slots = sa32(a.sm_slot) + 8u * (CL_MAXC * par);
            if (!(c.flags & CF_LOST)) {
                if (lane == 0) mb_expect(bar, a.C * 8);
                if (lane < a.C) st_async(remote(slots + 8u * c.rank, lane), as_bits(tot), remote(bar, lane));
                mb_wait(bar, (c.nred >> 1) & 1, c.watch, c.flags);
            }
            __syncwarp();
            V y{};
            if (lane < a.C) y = as_acc(sp<const double>(a.sm_slot)[CL_MAXC * par + lane], V{});
            tot = comb(y);
        }
    }
    c.nred++;
    return tot;
}

// Cluster barrier at which every block learns whether a wait ran out in any.  Blocks may disagree on
// whether the solve goes on only after such a wait, and its block has said so here by then: all take
// part in the same barriers, and none leaves while others may reach its shared memory.  turn alternates.
template <bool MULTI> __device__ __forceinline__ bool agree(const ClusterArgs &a, ClWatch *w, int tid, int turn)
{
    __syncthreads();                                         // the block's waits are over
    if constexpr (!MULTI) return false;
    if (tid < a.C && has_failed(w))
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote(sptr(&w->any[turn]), tid)), "r"(1) : "memory");
    __syncwarp();
    cluster_sync_all();
    return *(volatile int *)&w->any[turn] != 0;
}

// shared scalars of the solve, written by thread 0 (V: f2 or double)
template <class T, class V> struct ClScal { V rz0, rz; T alpha, beta; double rmax; int inner_done; };

// (float)(a / b) of two totals, the bits of the FP64 division: the quotient in df64 (about 2^-44) decides
// the rounding unless it lies next to a tie, where FP64 does (a division there is a chain of about
// twenty instructions of 64 cycles each).
__device__ __forceinline__ double ratio_f(double a, double b) { return a / b; }
__device__ __forceinline__ float ratio_f(f2 a, f2 b)
{
    const float q0 = a.h / b.h;
    const float r = fmaf(-q0, b.h, a.h) + fmaf(-q0, b.l, a.l);   // remainder (its leading part is exact)
    const float q1 = r / b.h;
    const f2 q = two_sum(q0, q1);
    // half an ulp of q.h, and the distance of the low part from it
    const float up = __int_as_float(__float_as_int(q.h) + 1), half = 0.5f * fabsf(up - q.h);
    if (fabsf(fabsf(q.l) - half) > 1e-3f * half && fabsf(fabsf(q.l) - 0.5f * half) > 1e-3f * half && fabsf(q.h) > 1e-30f && fabsf(q.h) < 1e30f) return q.h;
    return (float)(df_to_d(a) / df_to_d(b));
}
__device__ __forceinline__ bool positive(f2 v) { return v.h > 0.f; }   // (a normalised pair has its high word's sign)
__device__ __forceinline__ bool positive(double v) { return v > 0.0; }
// v > tol w for positive totals: by the high words unless they nearly meet
__device__ __forceinline__ bool above(f2 v, double tol, float tolf, f2 w)
{
    const float t = tolf * w.h;
    if (v.h > 1.001f * t) return true;
    if (v.h < 0.999f * t) return false;
    return df_to_d(v) > tol * df_to_d(w);
}
__device__ __forceinline__ bool above(double v, double tol, float, double w) { return v > tol * w; }

template <class T> struct Dot;
template <> struct Dot<float> {
    f2 v{0.f, 0.f};
    __device__ __forceinline__ void add(float a0, float b0, float a1, float b1) { v = df_add_f(v, fmaf(a0, b0, a1 * b1)); }
};
template <> struct Dot<double> {
    double v = 0.0;
    __device__ __forceinline__ void add(double a0, double b0, double a1, double b1) { v = fma(a0, b0, fma(a1, b1, v)); }
};
// ------------------------------------------------------------------------------------ outer residual
// r = b - A x on the block's cells (df64 as k_outer_residual_mx, rounded to FP32); returns max |r|
template <int B>
__device__ __forceinline__ float outer_res(const ClusterArgs &a, const SolveArgs &sa, const Ctx<float, 0> &c, long long off, int bx, int by,
                                           unsigned int lo, unsigned int hi, unsigned int fl, float (&r)[B][B])
{
    float rmax = 0.f;
    const bool act = (c.flags & CF_ACT) != 0;
    const long long at = off + (long long)by * B * a.P + bx * B;
    const float *xh = sa.xh + at, *xl = sa.xl + at;
    float h[B + 2][B], l[B + 2][B];
#pragma unroll
    for (int q = 0; q < B + 2; ++q) {
        const int j = by * B - 1 + q;
#pragma unroll
        for (int i = 0; i < B; ++i) h[q][i] = l[q][i] = 0.f;
        if (act && j >= 0 && j < sa.ny) {
            ldg_row(xh + (long long)(q - 1) * a.P, h[q]);
            ldg_row(xl + (long long)(q - 1) * a.P, l[q]);
        }
    }
    const f2 cx{sa.mc.cxh, sa.mc.cxl}, cy{sa.mc.cyh, sa.mc.cyl};
    // differences across faces: an open face's two cells take it with opposite signs (exactly), a
    // closed one gives zero; a difference is normalised, so its sum with zero is itself
    const f2 z{0.f, 0.f};
    auto neg = [](f2 v) { return f2{-v.h, -v.l}; };
    f2 dS[B];
#pragma unroll
    for (int i = 0; i < B; ++i) {
        const int s4 = 4 * i;
        dS[i] = (lo >> s4 & 4u) ? df_sub(f2{h[1][i], l[1][i]}, f2{h[0][i], l[0][i]}) : z;
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
        f2 W{__shfl_up_sync(0xffffffffu, h[q + 1][B - 1], 1), __shfl_up_sync(0xffffffffu, l[q + 1][B - 1], 1)};
        f2 E{__shfl_down_sync(0xffffffffu, h[q + 1][0], 1), __shfl_down_sync(0xffffffffu, l[q + 1][0], 1)};
        float bh[B], bl[B];
#pragma unroll
        for (int i = 0; i < B; ++i) bh[i] = bl[i] = 0.f;
        if (act) {
            ldg_row(sa.bh + at + (long long)q * a.P, bh);
            ldg_row(sa.bl + at + (long long)q * a.P, bl);
            if (!(c.flags & CF_WLANE)) W = bx > 0 ? f2{__ldcg(xh + (long long)q * a.P - 1), __ldcg(xl + (long long)q * a.P - 1)} : f2{0.f, 0.f};
            if (!(c.flags & CF_ELANE)) E = bx * B + B < sa.nx ? f2{__ldcg(xh + (long long)q * a.P + B), __ldcg(xl + (long long)q * a.P + B)} : f2{0.f, 0.f};
        }
        f2 dW = z;
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int s4 = 4 * (q * B + i);
            const unsigned int o = (s4 < 32 ? lo >> (s4 & 31) : hi >> (s4 & 31)) & 15u;
            const f2 xc{h[q + 1][i], l[q + 1][i]};
            const f2 xE = i < B - 1 ? f2{h[q + 1][i < B - 1 ? i + 1 : 0], l[q + 1][i < B - 1 ? i + 1 : 0]} : E;
            if (i == 0) dW = (o & 1u) ? df_sub(xc, W) : z;
            const f2 dE = (o & 2u) ? df_sub(xc, xE) : z;
            const f2 dN = (o & 8u) ? df_sub(xc, f2{h[q + 2][i], l[q + 2][i]}) : z;
            const f2 ax = df_add(df_mul(df_add(dW, dE), cx), df_mul(df_add(dS[i], dN), cy));
            dW = neg(dE);
            dS[i] = neg(dN);
            const float rv = df_sub(f2{bh[i], bl[i]}, ax).h;
            r[q][i] = (fl >> (q * B + i) & 1u) ? rv : 0.f;
            rmax = fmaxf(rmax, fabsf(r[q][i]));
        }
    }
    return rmax;
}
template <int B>
__device__ __forceinline__ double outer_res(const ClusterArgs &a, const SolveArgs &sa, const Ctx<double, 0> &c, long long off, int bx, int by,
                                            unsigned int lo, unsigned int hi, unsigned int fl, double (&r)[B][B])
{
    double rmax = 0.0;
    const bool act = (c.flags & CF_ACT) != 0;
    const long long at = off + (long long)by * B * a.P + bx * B;
    const double *x = sa.x + at;
    double h[B + 2][B];
#pragma unroll
    for (int q = 0; q < B + 2; ++q) {
        const int j = by * B - 1 + q;
#pragma unroll
        for (int i = 0; i < B; ++i) h[q][i] = 0.0;
        if (act && j >= 0 && j < sa.ny) ldg_row(x + (long long)(q - 1) * a.P, h[q]);
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
        double W = __shfl_up_sync(0xffffffffu, h[q + 1][B - 1], 1), E = __shfl_down_sync(0xffffffffu, h[q + 1][0], 1);
        double bv[B];
#pragma unroll
        for (int i = 0; i < B; ++i) bv[i] = 0.0;
        if (act) {
            ldg_row(sa.b + at + (long long)q * a.P, bv);
            if (!(c.flags & CF_WLANE)) W = bx > 0 ? __ldcg(x + (long long)q * a.P - 1) : 0.0;
            if (!(c.flags & CF_ELANE)) E = bx * B + B < sa.nx ? __ldcg(x + (long long)q * a.P + B) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int s4 = 4 * (q * B + i);
            const unsigned int o = (s4 < 32 ? lo >> (s4 & 31) : hi >> (s4 & 31)) & 15u;
            const double xc = h[q + 1][i];
            const double xW = i > 0 ? h[q + 1][i > 0 ? i - 1 : 0] : W, xE = i < B - 1 ? h[q + 1][i < B - 1 ? i + 1 : 0] : E;
            const double cW = (o & 1u) ? sa.cxd : 0.0, cE = (o & 2u) ? sa.cxd : 0.0, cS = (o & 4u) ? sa.cyd : 0.0, cN = (o & 8u) ? sa.cyd : 0.0;
            double ax = (((cW + cE) + cS) + cN) * xc;
            ax = fma(-cW, xW, ax);
            ax = fma(-cE, xE, ax);
            ax = fma(-cS, h[q][i], ax);
            ax = fma(-cN, h[q + 2][i], ax);
            r[q][i] = (fl >> (q * B + i) & 1u) ? bv[i] - ax : 0.0;
            rmax = fmax(rmax, fabs(r[q][i]));
        }
    }
    return rmax;
}

// Fluid sum of x (its high words), in the order of k_outer_residual_mx and res_finish_member: warps of
// 64 columns x 4 rows, blocks of eight of them, then the blocks' partials by one warp.  The mean it
// gives enters the pressure and the next guess, and cancels almost to zero, so its bits depend on the
// order; mixed handles sum in the same order on either solve path.
template <bool MULTI>
__device__ double fluid_sum_mx(const ClusterArgs &a, const SolveArgs &sa, Ctx<float, 0> &c, long long off, int turn, bool *failed)
{
    const int gx = (sa.nx + 63) / 64, gy = (sa.ny + 31) / 32, nb = gx * gy;
    const int lane = c.tid & 31, w = c.tid >> 5, nw = (int)blockDim.x >> 5;
    f2 *unit = sp<f2>(a.sm_xs);        // [blocks of this rank][8]
    const int mine = (nb - c.rank + a.C - 1) / a.C;
    // four units of a warp in flight
    for (int u0 = w; u0 < 8 * mine; u0 += 4 * nw) {
        float2 xv[4][4];
        unsigned int fl[4][4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int u = u0 + v * nw, q = c.rank + (u >> 3) * a.C, bx = q % gx, by = q / gx, i = bx * 64 + 2 * lane;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int j = (by * 8 + (u & 7)) * 4 + r;
                fl[v][r] = 0u;
                xv[v][r] = make_float2(0.f, 0.f);
                if (u < 8 * mine && i < sa.nx && j < sa.ny) {
                    const long long at = (long long)j * a.P + i;
                    fl[v][r] = *reinterpret_cast<const unsigned short *>(sa.fluid + at);
                    xv[v][r] = __ldcg(reinterpret_cast<const float2 *>(sa.xh + off + at));
                }
            }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            f2 xs{0.f, 0.f};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if (fl[v][r] & 0xffu) xs = df_add_f(xs, xv[v][r].x);
                if (fl[v][r] >> 8) xs = df_add_f(xs, xv[v][r].y);
            }
            xs = warp_sum_df(xs);
            if (lane == 0 && u0 + v * nw < 8 * mine) unit[u0 + v * nw] = xs;
        }
    }
    __syncthreads();
    const int m = blockIdx.x / a.C;
    double *slots = sa.rc.part + ((long long)RS_XSUM * sa.rc.stride + m) * sa.rc.nblk;
    for (int t = w; t < mine; t += nw) {
        f2 v = lane < 8 ? unit[8 * t + lane] : f2{0.f, 0.f};
        v = warp_sum_df(v);
        if (lane == 0) *reinterpret_cast<float2 *>(slots + c.rank + t * a.C) = make_float2(v.h, v.l);
    }
    *failed = agree<MULTI>(a, c.watch, c.tid, turn);
    double tot = 0.0;
    if (c.rank == 0 && w == 0) {
        f2 xs{0.f, 0.f};
        for (int q = lane; q < nb; q += 32) {
            const float2 v = __ldcg(reinterpret_cast<const float2 *>(slots + q));
            xs = df_add(xs, f2{v.x, v.y});
        }
        xs = warp_sum_df(xs);
        if (lane == 0) tot = df_to_d(xs);
    }
    return tot;
}

// ------------------------------------------------------------------------------------ the kernel
// Threads per block at most: the registers of 640 threads fit twice 48; a mixed 4 x 4 block keeps its
// iterate and right-hand side (32 values) with one level's conductances (16) in 96 registers.
// FP64 2 x 2 blocks: 152 registers without spills up to 192 threads, with which two blocks still share an SM;
// beyond, 128 (512 threads), for the same reason.  (At 80 registers and 768 threads 400 bytes per thread spilled: 128 x 64,
// one member at a time: 51.7 ms, now 43.3 ms; 176 x 80, 17 members: 10.4 ms, with 152 registers and one block per
// SM 13.7 ms, with 128 registers 10.0 ms.)
constexpr int CL_FEW_THREADS = 192, CL_FEW_BOUND = 384;
// Mixed 4 x 4 blocks up to 512 threads: 128 registers where an SM holds one block anyway (more than 320 threads,
// or 112 KB; 96 registers spill 460 bytes per thread): 256 x 128, 33 members 7.31 -> 6.56 ms, 5 members 2.96 -> 2.70 ms.
constexpr int CL_MID_BOUND = 512;
template <class T, int B> struct ClLimit { static constexpr int threads = B == 2 ? (sizeof(T) == 4 ? 768 : 512) : sizeof(T) == 4 ? 640 : 352; };

template <class T, int B, bool FIRST, bool MULTI, int BOUND>
__global__ void __launch_bounds__(BOUND, 1) k_cluster(const __grid_constant__ ClusterArgs a, const __grid_constant__ SolveArgs sa)
{
    __shared__ ClScal<T, decltype(Dot<T>::v)> sc;
    __shared__ ClWatch watch;
    const int rank = MULTI ? cluster_rank() : 0;
    const int m = blockIdx.x / a.C, tid = threadIdx.x;
    if (sa.ctl[m].outer_done) return;                        // every block of the cluster reads the same word
    if (sa.mode == 1 && sa.inner_guard && sa.ctl[m].inner_done) return;
    const long long off = (long long)m * a.S;
    if (tid == 0) {
        watch = ClWatch{0, sa.wait_limit, {0, 0}};
        for (int q = 0; q < 8; ++q) mb_init(sa32(8 * q), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // zero the planes: solid blocks and the domain's surroundings stay zero
    {
        const int beg = a.st[0].plane[0] >> 4, end = a.sm_p >> 4;
        for (int q = beg + tid; q < end; q += blockDim.x) sp<uint4>(0)[q] = make_uint4(0u, 0u, 0u, 0u);
    }
    T *lut = sp<T>(a.sm_lut);
    const T cx = sizeof(T) == 4 ? (T)sa.cxf : (T)sa.cxd, cy = sizeof(T) == 4 ? (T)sa.cyf : (T)sa.cyd;
    if (rank == 0)
        for (int q = tid; q < (int)(sizeof(a.st) / 4); q += blockDim.x) sp<int>(a.sm_st)[q] = reinterpret_cast<const int *>(a.st)[q];
    // conductance tables, and the gathered stages' fluid bits
    for (int s = sizeof(T) == 4 ? 0 : 1; s < (rank == 0 ? a.nst : 1); ++s) {
        const ClStageArgs &st = a.st[s];
        for (int k = 0; k < st.nlev; ++k) {
            const int b = st.B >> k, n = (2 * b * (b + 1) + b * b) * st.nrec[k];
            for (int q = tid; q < n; q += blockDim.x) sp<T>(st.simg[k])[q] = reinterpret_cast<const T *>(st.img[k])[q];
        }
        if (s > 0)
            for (int q = tid; q < st.ni; q += blockDim.x) sp<int>(st.sfm)[q] = st.fm[q];
    }
    if (FIRST && tid < 16) {
        const unsigned int q = tid;
        const T d = ((q & 1u) ? cx : (T)0) + ((q & 2u) ? cx : (T)0) + ((q & 4u) ? cy : (T)0) + ((q & 8u) ? cy : (T)0);
        lut[q] = d;
        lut[16 + q] = (d != (T)0) ? (T)1 / d : (T)0;
    }
    Ctx<T, 0> c;
    c.tid = tid; c.rank = rank; c.id = 0; c.nt = a.nt; c.watch = &watch;
    c.n = c.gat = c.nred = 0;
    const int4 rec = a.rec[rank * a.nt + tid];
    const int bx = rec.x & 0xffff, by = (rec.x >> 16) & 0xffff;
    c.flags = rec.y & 0xffff;
    const unsigned int fl = (unsigned int)rec.y >> 16;
    const bool act = (c.flags & CF_ACT) != 0;
    c.fm = act ? a.st[0].fm[rank * a.nt + tid] : 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) c.kind[k] = (B >> k) && (k > 0 || !FIRST) ? a.st[0].kind[k][rank * a.nt + tid] : 0;
    {
        const ClSlab s = a.slab[rank];
        c.rxS = s.rxS; c.rxN = s.rxN;
        if constexpr (MULTI) {
            // a push to the south lands in the neighbour's north halo and the other way round
            c.rbarS = remote(sa32(BAR_N), rank > 0 ? rank - 1 : 0);
            c.rbarN = remote(sa32(BAR_S), rank + 1 < a.C ? rank + 1 : rank);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int b = B >> k;
            if (b < 1) break;
            c.pitch[k] = act ? (s.wb * b + 2 * CL_PAD) * (int)sizeof(T) : 128;
            c.own[k] = act ? a.st[0].plane[k] + ((by - s.rb0) * b + 1) * c.pitch[k] + (CL_PAD + (bx - s.cb0) * b) * (int)sizeof(T) : a.sm_idle + 128 + 32;
            if constexpr (MULTI) {
                c.pushS[k] = c.pushN[k] = 0u;
                const unsigned int pl = sa32(a.st[0].plane[k]);
                if (c.flags & CF_PUSH_S) {
                    const ClSlab t = a.slab[rank - 1];
                    c.pushS[k] = remote(pl, rank - 1) + (unsigned int)sizeof(T) * ((t.hb * b + 1) * (t.wb * b + 2 * CL_PAD) + CL_PAD + (bx - t.cb0) * b);
                }
                if (c.flags & CF_PUSH_N) {
                    const ClSlab t = a.slab[rank + 1];
                    c.pushN[k] = remote(pl, rank + 1) + (unsigned int)sizeof(T) * (CL_PAD + (bx - t.cb0) * b);
                }
            }
        }
    }
    if constexpr (MULTI) cluster_sync_all();
    else __syncthreads();

    const long long at = off + (long long)by * B * a.P + bx * B;   // the block's first cell
    T f[B][B], e[B][B];
    bool failed = false;

    if constexpr (!FIRST) {
        // mode 1: one V-cycle of the levels from la
#pragma unroll
        for (int r = 0; r < B; ++r) {
#pragma unroll
            for (int i = 0; i < B; ++i) f[r][i] = (T)0;
            if (act) ldg_row(reinterpret_cast<const T *>(sa.f) + at + (long long)r * a.P, f[r]);
        }
        vlevel<T, B, MULTI>(a, c, 0, f, e);
        if (act) {
#pragma unroll
            for (int r = 0; r < B; ++r) st_row(reinterpret_cast<T *>(sa.e) + at + (long long)r * a.P, e[r]);
        }
        failed = agree<MULTI>(a, &watch, tid, 0);
    } else {
        Open<T, B> q;
        q.cx = cx; q.cy = cy; q.lut = lut;
        q.lo = (unsigned int)rec.z; q.hi = (unsigned int)rec.w;
        q.all = __all_sync(0xffffffffu, q.lo == (B == 4 ? 0xffffffffu : 0xffffu) && (B == 2 || q.hi == 0xffffffffu));
        unsigned int om = 0u;                                // cells with an open face (prolongation)
#pragma unroll
        for (int r = 0; r < B; ++r)
#pragma unroll
            for (int i = 0; i < B; ++i) om |= (q.bits(r, i) ? 1u : 0u) << (r * B + i);
        T *pst = sp<T>(a.sm_p);         // search direction, [row][thread][B]
        T *acc = reinterpret_cast<T *>(sa.acc) + at;
        int outer_its = 0, inner_its = 0;
        bool done = false;
        bool closed = false;                                 // the loop ended at a residual
        double rmax_d = 0.0;
        int o = sa.first_o;
        for (;; ++o) {
            {
                const auto rm = outer_res<B>(a, sa, c, off, bx, by, q.lo, q.hi, fl, f);
                const double t = cluster_total<T, double, MULTI, true>(a, c, (double)rm);
                if (tid == 0) { sc.rmax = t; sc.inner_done = 0; }
                __syncthreads();
                rmax_d = sc.rmax;
            }
            done = rmax_d <= sa.rtol_abs;
            if (!done && (sa.count_last || o < sa.max_outer)) ++outer_its;
            closed = done || o == sa.max_outer;
            if (closed) break;
            // ---- one refinement: V-cycle-preconditioned CG on A e = r, then x += e
            bool stop = false, have_acc = false;
            for (int k = 0; k <= sa.max_inner; ++k) {
                if (k == sa.max_inner) break;
                if (k == 0 || !stop) {
                    // z = M r
                    descend<T, B, 0, MULTI>(c, 0, a.nu[0][0], q, f, e);
                    {
                        T res[B][B], fc[B / 2][B / 2], ec[B / 2][B / 2];
                        residual<T, B, 0>(c, 0, q, 0, f, e, res);
#pragma unroll
                        for (int r = 0; r < B / 2; ++r)
#pragma unroll
                            for (int i = 0; i < B / 2; ++i)
                                fc[r][i] = sum4(res[2 * r][2 * i], res[2 * r][2 * i + 1], res[2 * r + 1][2 * i], res[2 * r + 1][2 * i + 1], 0);
                        vlevel<T, B / 2, MULTI>(a, c, 1, fc, ec);
                        prolong<T, B>(om, ec, e);
                    }
                    ascend<T, B, 0, MULTI>(c, 0, a.nu[0][1], q, f, e);
                    Dot<T> d;
#pragma unroll
                    for (int r = 0; r < B; ++r)
#pragma unroll
                        for (int i = 0; i < B; i += 2) d.add(f[r][i], e[r][i], f[r][i + 1], e[r][i + 1]);
                    const auto t = cluster_total<T, decltype(d.v), MULTI, false>(a, c, d.v);
                    if (tid == 0) {
                        if (k == 0) {
                            sc.rz0 = t;
                            if (!positive(t)) sc.inner_done = 1;
                        } else {
                            sc.beta = ratio_f(t, sc.rz);
                            if (!above(t, sa.inner_rtol2, (float)sa.inner_rtol2, sc.rz0)) sc.inner_done = 1;
                        }
                        sc.rz = t;
                    }
                    __syncthreads();
                    stop = sc.inner_done != 0;
                }
                const bool last = k + 1 == sa.max_inner;
                if (stop && !last) continue;                 // only the final update of x is left
                T ap = (T)0;
                if (!stop) {
                    // p = z + beta p, q = A p, p.q
                    const T bt = sc.beta;
#pragma unroll
                    for (int r = 0; r < B; ++r) {
                        if (k > 0) {
                            T pv[B];
                            ld_row(pst + (r * a.nt + tid) * B, pv);
#pragma unroll
                            for (int i = 0; i < B; ++i) e[r][i] = fma_(bt, pv[i], e[r][i]);
                        }
                        st_row(pst + (r * a.nt + tid) * B, e[r]);
                    }
                    exchange<T, B, 0, MULTI>(c, 0, e);
                    T qv[B][B];
                    Dot<T> d;
                    {
                        T s[B], n[B];
                        rows_sn<T, B, 0>(c, 0, s, n);
#pragma unroll
                        for (int r = 0; r < B; ++r) {
                            const T wv = west<T, B, 0>(c, 0, e, r), ev = east<T, B, 0>(c, 0, e, r);
#pragma unroll
                            for (int i = 0; i < B; ++i) {
                                const T w = i > 0 ? e[r][i > 0 ? i - 1 : 0] : wv, oo = i < B - 1 ? e[r][i < B - 1 ? i + 1 : 0] : ev;
                                const T ss = r > 0 ? e[r > 0 ? r - 1 : 0][i] : s[i], nn = r < B - 1 ? e[r < B - 1 ? r + 1 : 0][i] : n[i];
                                const unsigned int t = q.bits(r, i);
                                qv[r][i] = t ? fma_(-cy, ss + nn, fma_(lut[t], e[r][i], -(cx * (w + oo)))) : (T)0;
                            }
#pragma unroll
                            for (int i = 0; i < B; i += 2) d.add(e[r][i], qv[r][i], e[r][i + 1], qv[r][i + 1]);
                        }
                    }
                    const auto t = cluster_total<T, decltype(d.v), MULTI, false>(a, c, d.v);
                    if (tid == 0) {
                        sc.alpha = ratio_f(sc.rz, t);
                        if (!positive(t)) sc.inner_done = 1; // breakdown: stop this member's inner loop
                    }
                    __syncthreads();
                    stop = sc.inner_done != 0;
                    ap = sc.alpha;
                    if (!stop) {
                        ++inner_its;
                        if (!last) {
#pragma unroll
                            for (int r = 0; r < B; ++r)
#pragma unroll
                                for (int i = 0; i < B; ++i) f[r][i] = fma_(-ap, qv[r][i], f[r][i]);
                        }
                    }
                }
                const bool moving = !stop;
                if (last) {
                    // x += e + alpha p
                    if (act) {
                        // (f is formed anew by the next residual: its registers hold e's increment)
#pragma unroll
                        for (int r = 0; r < B; ++r) {
#pragma unroll
                            for (int i = 0; i < B; ++i) f[r][i] = (T)0;
                            if (have_acc) ldg_row(acc + (long long)r * a.P, f[r]);
                        }
#pragma unroll
                        for (int r = 0; r < B; ++r) {
                            T (&d)[B] = f[r];
                            if constexpr (sizeof(T) == 4) {
                                float h[B], l[B];
                                float *xh = sa.xh + at + (long long)r * a.P, *xl = sa.xl + at + (long long)r * a.P;
                                ldg_row(xh, h);
                                ldg_row(xl, l);
                                if (moving) {
#pragma unroll
                                    for (int i = 0; i < B; ++i) d[i] = fma_(ap, e[r][i], d[i]);
                                }
#pragma unroll
                                for (int i = 0; i < B; ++i)
                                    if (d[i] != 0.f) {
                                        const f2 s = df_add_f(f2{h[i], l[i]}, d[i]);
                                        h[i] = s.h;
                                        l[i] = s.l;
                                    }
                                st_row(xh, h);
                                st_row(xl, l);
                            } else {
                                if (moving) {
#pragma unroll
                                    for (int i = 0; i < B; ++i) d[i] = fma_(ap, e[r][i], d[i]);
                                }
                                double h[B];
                                double *x = sa.x + at + (long long)r * a.P;
                                ldg_row(x, h);
#pragma unroll
                                for (int i = 0; i < B; ++i)
                                    if (fl >> (r * B + i) & 1u) h[i] += d[i];
                                st_row(x, h);
                            }
                        }
                    }
                } else if (moving) {
                    // e += alpha p
                    if (act) {
#pragma unroll
                        for (int r = 0; r < B; ++r) {
                            T d[B];
#pragma unroll
                            for (int i = 0; i < B; ++i) d[i] = (T)0;
                            if (have_acc) ldg_row(acc + (long long)r * a.P, d);
#pragma unroll
                            for (int i = 0; i < B; ++i) d[i] = fma_(ap, e[r][i], d[i]);
                            st_row(acc + (long long)r * a.P, d);
                        }
                    }
                    have_acc = true;
                }
            }
            failed = agree<MULTI>(a, &watch, tid, o & 1);    // x of every block before the next residual reads it
            if (failed || sa.one) break;
        }
        // totals and flags of the member (the fluid sum of x is its mean's numerator)
        double xs = 0.0;
        if (!closed) {
        } else if constexpr (sizeof(T) == 4) {
            xs = fluid_sum_mx<MULTI>(a, sa, c, off, o & 1, &failed);
        } else {
            double v = 0.0;
            if (act) {
#pragma unroll
                for (int r = 0; r < B; ++r) {
                    double h[B];
                    ldg_row(sa.x + at + (long long)r * a.P, h);
#pragma unroll
                    for (int i = 0; i < B; ++i)
                        if (fl >> (r * B + i) & 1u) v += h[i];
                }
            }
            xs = cluster_total<T, double, MULTI, false>(a, c, v);
            failed = agree<MULTI>(a, &watch, tid, o & 1);
        }
        if (rank == 0 && tid == 0) {
            MemberRed &red = sa.rc.red[m];
            if (closed || failed) {
                red.val[RS_RMAX] = failed ? 1e300 : rmax_d;
                red.val[RS_XSUM] = failed ? 0.0 : xs;
            }
            MemberCtl &mc = sa.ctl[m];
            mc.outer_done = done && !failed;
            mc.inner_done = done && !failed;
            mc.outer_its += outer_its;
            mc.inner_its += inner_its;
        }
    }
    if (failed) {
        // a wait ran out: the member counts as unconverged.  Stores that nobody waited for may still be on
        // their way; no block sends more, and a tenth of a millisecond is two hundred times their latency.
        if (rank == 0 && tid == 0) atomicOr(&sa.ctl[m].status, ENVAR_ST_DIVERGENCE);
#pragma unroll 1
        for (int k = 0; k < 16; ++k) __nanosleep(8000);
        cluster_sync_all();
    }
    // (otherwise the last agree ended all access to other blocks' shared memory: no barrier before the exit)
}

// ------------------------------------------------------------------------------------ plan (host)
struct ClusterPlan {
    ClusterArgs a{};
    int threads = 0;
    size_t smem = 0;
    bool multi = false;
};

// smoothing factors of a level with explicit conductances, from the diagonal sums the host put in
// their place: the tiled smoothers' 1 / d, or the coarse block's fast reciprocal
__global__ void k_cluster_factor(float *v, long long n, int fast)
{
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const float d = v[q];
        v[q] = d != 0.f ? (fast ? __fdividef(1.f, d) : 1.f / d) : 0.f;
    }
}
__global__ void k_cluster_factor(double *v, long long n, int)
{
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const double d = v[q];
        v[q] = d != 0.0 ? 1.0 / d : 0.0;
    }
}

// Slabs of consecutive block rows for C thread blocks: the smallest largest cost, a slab's cost being
// the larger of its threads and of its border plane (bounding box of its fluid blocks), each as a
// fraction of what a block may have.  first[k]: first row of slab k.
static bool cut_rows(const std::vector<int> &cnt, const std::vector<int> &x0, const std::vector<int> &x1, int C, int B, int max_threads,
                     double max_plane_cells, std::vector<int> *first)
{
    const int n = (int)cnt.size();
    if (n < C) return false;
    const double none = 1e30;
    std::vector<std::vector<double>> best(C + 1, std::vector<double>(n + 1, none));
    std::vector<std::vector<int>> from(C + 1, std::vector<int>(n + 1, -1));
    best[0][0] = 0.0;
    for (int j = 1; j <= n; ++j) {
        int c = 0, lo = 1 << 30, hi = -1;
        for (int i = j - 1; i >= 0; --i) {                   // slab of rows i .. j-1
            c += cnt[i];
            lo = std::min(lo, x0[i]);
            hi = std::max(hi, x1[i]);
            if (c > max_threads) break;
            if (hi < lo) continue;
            const double plane = ((double)(hi - lo + 1) * B + 2 * CL_PAD) * ((j - i) * B + 2);
            const double cost = std::max((double)c / max_threads, plane / max_plane_cells);
            for (int k = 1; k <= C; ++k) {
                const double v = std::max(best[k - 1][i], cost);
                if (best[k - 1][i] < none && v < best[k][j]) { best[k][j] = v; from[k][j] = i; }
            }
        }
    }
    if (!(best[C][n] <= 1.0)) return false;
    first->assign(C, 0);
    for (int k = C, j = n; k > 0; --k) { j = from[k][j]; (*first)[k - 1] = j; }
    return true;
}

// The B x B blocks of a level that hold fluid, and each block row's count and extent.
struct ClBlocks {
    int B, bw, bh, nact = 0;
    std::vector<uint8_t> act;
    std::vector<int> cnt, x0, x1;
    ClBlocks(const ClusterHostLevel &L, int B_) : B(B_), bw(L.nx / B_), bh(L.ny / B_)
    {
        act.assign((size_t)bw * bh, 0);
        cnt.assign(bh, 0); x0.assign(bh, 1 << 30); x1.assign(bh, -1);
        // the block's cells of a row are a word (a copy of known size: 512 x 256, both B, 0.69 -> 0.05 ms)
        auto mark = [&](auto word) {
            for (int j = 0; j < bh * B; ++j) {
                const uint8_t *f = L.F + (size_t)j * L.P;
                uint8_t *q = &act[(size_t)(j / B) * bw];
                for (int x = 0; x < bw; ++x) {
                    std::memcpy(&word, f + x * sizeof(word), sizeof(word));
                    q[x] |= word != 0;
                }
            }
        };
        if (B == 4) mark((uint32_t)0);
        else mark((uint16_t)0);
        for (int y = 0; y < bh; ++y)
            for (int x = 0; x < bw; ++x)
                if (act[(size_t)y * bw + x]) { ++cnt[y]; x0[y] = std::min(x0[y], x); x1[y] = x; }
        for (int c : cnt) nact += c;
    }
    bool operator()(int x, int y) const { return x >= 0 && y >= 0 && x < bw && y < bh && act[(size_t)y * bw + x]; }
};

template <class T> static cudaError_t dispatch(const ClusterPlan &p, const SolveArgs &sa, int M, cudaStream_t st, bool query, int *active);

// Build the plan for the levels from la with B x B blocks on C thread blocks, its tables uploaded through `alloc`
// once nothing else can fail; nullptr when the grid does not fit the scheme or no such cluster is resident.
template <class T>
static ClusterPlan *make_plan(const ClusterHostLevel *hl, int nlev, int ncoarse, int la, const ClBlocks &bl, int C, const ClusterAlloc &alloc)
{
    const int B = bl.B, nloc = B == 4 ? 3 : 2, bw = bl.bw, bh = bl.bh;
    if (la + nloc >= nlev) return nullptr;                   // the coarsest level is in a gathered stage
    const ClusterHostLevel &L = hl[la];
    if (L.nx % B || L.ny % B || bw > 32767 || bh > 32767) return nullptr;
    // No kernel for these two: a level 1 that one block could hold belongs to a grid that runs whole in a cluster, and FP64
    // grids of one block run on 2 x 2 blocks of cells (no grid from 16 x 16 to 1400 x 900 in steps of 16, in four boxes, gets here
    // otherwise).
    if (C == 1 && (la > 0 || (sizeof(T) == 8 && B == 4))) return nullptr;
    const std::vector<int> &cnt = bl.cnt, &x0 = bl.x0, &x1 = bl.x1;
    const int nact = bl.nact, limit = B == 4 ? ClLimit<T, 4>::threads : ClLimit<T, 2>::threads;
    std::vector<int> first;
    if (nact > limit * C || !cut_rows(cnt, x0, x1, C, B, limit, 96.0 * 1024 / sizeof(T), &first)) return nullptr;
    auto active = [&](int x, int y) { return bl(x, y); };
    int most = 1;
    for (int k = 0; k < C; ++k) {
        int c = 0;
        for (int r = first[k]; r < (k + 1 < C ? first[k + 1] : bh); ++r) c += cnt[r];
        most = std::max(most, c);
    }
    const int nt = round_up(most, 32);
    ClusterPlan *P = new ClusterPlan();
    ClusterArgs &a = P->a;
    a.C = C; a.nt = nt; a.la = la; a.nact = nact;
    a.P = L.P; a.S = (long long)(L.ny + 1) * L.P;
    P->multi = C > 1;
    auto fail = [&]() -> ClusterPlan * { delete P; return nullptr; };
    // ---- stages
    int l = la + nloc, ns = 1;
    a.st[0].B = B; a.st[0].nlev = nloc; a.st[0].l0 = la; a.st[0].bw = bw; a.st[0].bh = bh; a.st[0].nt = nt;
    if (hl[l].nx * 2 != bw || hl[l].ny * 2 != bh) return fail();
    while (l < nlev) {
        if (ns >= CL_STAGES) return fail();
        const int left = nlev - l;
        const int q = (left >= 2 && hl[l].nx % 2 == 0 && hl[l].ny % 2 == 0) ? 2 : 1;
        ClStageArgs &s = a.st[ns];
        s.B = q; s.nlev = q; s.l0 = l; s.bw = hl[l].nx / q; s.bh = hl[l].ny / q;
        s.nt = round_up(s.bw * s.bh, 32);
        s.rbw = 0xffffffffu / (unsigned int)s.bw + 1u;
        s.ni = s.nt;
        if (la > 0 && ns == 1 && s.nlev == 1 && l + 1 == nlev && s.nt > nt && s.nt <= 4 * nt) {
            s.wide = 1;
            s.nt = nt;
        }
        if (s.nt > nt || s.bw < 2) return fail();
        l += s.nlev;
        ++ns;
    }
    a.nst = ns;
    for (int s = 0; s < ns; ++s)
        for (int k = 0; k < a.st[s].nlev; ++k) {
            const int lev = a.st[s].l0 + k;
            // the tiled smoothers with coded conductances (and the first level's) add row pairs
            a.st[s].seq[k] = lev >= ncoarse || (lev > 0 && !hl[lev].coded);
        }
    // ---- slabs
    for (int k = 0; k < C; ++k) {
        ClSlab &s = a.slab[k];
        s.rb0 = first[k];
        s.hb = (k + 1 < C ? first[k + 1] : bh) - s.rb0;
        int x0 = bw, x1 = -1;
        for (int y = s.rb0; y < s.rb0 + s.hb; ++y)
            for (int x = 0; x < bw; ++x)
                if (active(x, y)) { x0 = std::min(x0, x); x1 = std::max(x1, x); }
        if (x1 < 0) return fail();
        s.cb0 = x0;
        s.wb = x1 - x0 + 1;
        s.rxS = s.rxN = 0;
        for (int x = 0; x < bw; ++x) {
            if (k > 0 && active(x, s.rb0) && active(x, s.rb0 - 1)) ++s.rxS;
            if (k + 1 < C && active(x, s.rb0 + s.hb - 1) && active(x, s.rb0 + s.hb)) ++s.rxN;
        }
    }
    // ---- per-thread records of stage 0 (blocks of a slab row by row; idle threads at the end)
    struct Th { int x, y; };
    std::vector<std::vector<Th>> th(C);
    for (int k = 0; k < C; ++k)
        for (int y = a.slab[k].rb0; y < a.slab[k].rb0 + a.slab[k].hb; ++y)
            for (int x = 0; x < bw; ++x)
                if (active(x, y)) th[k].push_back(Th{x, y});
    std::vector<int4> rec((size_t)C * nt, int4{0, 0, 0, 0});
    for (int k = 0; k < C; ++k) {
        const ClSlab &s = a.slab[k];
        for (size_t t = 0; t < th[k].size(); ++t) {
            const int x = th[k][t].x, y = th[k][t].y, lane = (int)t & 31;
            int fg = CF_ACT;
            if (lane > 0 && th[k][t - 1].x == x - 1 && th[k][t - 1].y == y) fg |= CF_WLANE;
            if (lane < 31 && t + 1 < th[k].size() && th[k][t + 1].x == x + 1 && th[k][t + 1].y == y) fg |= CF_ELANE;
            if (k > 0 && y == s.rb0 && active(x, y - 1)) fg |= CF_PUSH_S | CF_WAIT_S;
            if (k + 1 < C && y == s.rb0 + s.hb - 1 && active(x, y + 1)) fg |= CF_PUSH_N | CF_WAIT_N;
            if ((x ^ y) & 1) fg |= CF_PAR;
            unsigned int fl = 0;
            uint64_t ob = 0;
            for (int r = 0; r < B; ++r) {
                const size_t cc = (size_t)(y * B + r) * L.P + x * B;
                for (int i = 0; i < B; ++i) fl |= (L.F[cc + i] ? 1u : 0u) << (r * B + i);
                for (int i = 0; i < B && la == 0; ++i) ob |= (uint64_t)(L.open[cc + i] & 15) << (4 * (r * B + i));
            }
            rec[(size_t)k * nt + t] = int4{x | (y << 16), fg | (int)(fl << 16), (int)(unsigned int)ob, (int)(unsigned int)(ob >> 32)};
        }
    }
    // ---- per-level conductances, smoothing factors (their denominators, here) and fluid bits
    std::vector<T> table[CL_STAGES][3];
    std::vector<int> kind[3], fm[CL_STAGES];
    for (int s = 0; s < ns; ++s) {
        ClStageArgs &st = a.st[s];
        const int n = s == 0 ? C * nt : st.ni;
        fm[s].assign(n, 0);
        auto block = [&](int t, int *x, int *y) {
            if (s == 0) {
                const int4 q = rec[t];
                *x = q.x & 0xffff; *y = (q.x >> 16) & 0xffff;
                return (q.y & CF_ACT) != 0;
            }
            *x = t % st.bw; *y = t / st.bw;
            return t < st.bw * st.bh;
        };
        for (int k = 0; k < st.nlev; ++k) {
            const int b = st.B >> k, lev = st.l0 + k;
            const ClusterHostLevel &H = hl[lev];
            if (lev == 0) {                                  // uniform conductances: no image
                st.nrec[k] = 0;
                continue;
            }
            const int nc = 2 * b * (b + 1), nv = b * b, sh = b == 4 ? 0 : b == 2 ? 16 : 20;
            // the values of block (x, y), and its fluid bits
            auto record_b = [&](auto size, int x, int y, T *w, size_t stride) {
                constexpr int b = decltype(size)::value;     // (known when compiled: half the time)
                int bits = 0;
                const size_t at = (size_t)(y * b) * H.P + x * b;
                for (int r = 0; r < b; ++r)
                    for (int i = 0; i <= b; ++i, w += stride) *w = (T)H.cw[at + r * H.P + i];
                for (int r = 0; r <= b; ++r)
                    for (int i = 0; i < b; ++i, w += stride) *w = (T)H.cs[at + r * H.P + i];
                for (int r = 0; r < b; ++r)
                    for (int i = 0; i < b; ++i, w += stride) {
                        const size_t cc = at + r * H.P + i;
                        *w = (((T)H.cw[cc] + (T)H.cw[cc + 1]) + (T)H.cs[cc]) + (T)H.cs[cc + H.P];
                        bits |= (H.F[cc] ? 1 : 0) << (sh + r * b + i);
                    }
                return bits;
            };
            auto record = [&](int x, int y, T *w, size_t stride) {
                return b == 4 ? record_b(std::integral_constant<int, 4>(), x, y, w, stride)
                     : b == 2 ? record_b(std::integral_constant<int, 2>(), x, y, w, stride)
                              : record_b(std::integral_constant<int, 1>(), x, y, w, stride);
            };
            std::vector<T> im;
            size_t nr = n;
            if (s == 0) {                                    // equal records are one
                std::map<std::vector<T>, int> seen;
                std::vector<T> r((size_t)nc + nv, (T)0), last;
                kind[k].resize(n);
                for (int t = 0; t < n; ++t) {
                    int x, y;
                    if (block(t, &x, &y)) fm[s][t] |= record(x, y, r.data(), 1);
                    else r.assign(r.size(), (T)0);
                    if (t > 0 && r == last) {                // the neighbour's, mostly
                        kind[k][t] = kind[k][t - 1];
                        continue;
                    }
                    kind[k][t] = seen.emplace(r, (int)seen.size()).first->second;
                    last = r;
                }
                nr = seen.size();
                im.assign(r.size() * nr, (T)0);
                for (const auto &q : seen)
                    for (size_t w = 0; w < r.size(); ++w) im[w * nr + q.second] = q.first[w];
            } else {
                im.assign((size_t)(nc + nv) * n, (T)0);
                for (int t = 0; t < n; ++t) {
                    int x, y;
                    if (block(t, &x, &y)) fm[s][t] |= record(x, y, &im[t], n);
                }
            }
            st.nrec[k] = (int)nr;
            table[s][k] = std::move(im);
        }
    }
    // ---- shared memory
    size_t o = 64;                                           // eight barriers
    auto up16 = [](size_t b) { return (b + 15) & ~(size_t)15; };
    for (int k = 0; k < nloc; ++k) {
        size_t most_b = 0;
        const int b = B >> k;
        for (int r = 0; r < C; ++r)
            most_b = std::max(most_b, (size_t)(a.slab[r].wb * b + 2 * CL_PAD) * (a.slab[r].hb * b + 2));
        a.st[0].plane[k] = (int)o;
        o = up16(o + most_b * sizeof(T));
    }
    a.st[0].rp = (int)o;
    o = up16(o + (size_t)bw * bh * sizeof(T));
    for (int s = 1; s < ns; ++s) {
        for (int k = 0; k < a.st[s].nlev; ++k) {
            const int b = a.st[s].B >> k;
            a.st[s].pitch[k] = a.st[s].bw * b + 2 * CL_PAD + (a.st[s].bw * b) % 2;
            a.st[s].plane[k] = (int)o;
            o = up16(o + (size_t)a.st[s].pitch[k] * (a.st[s].bh * b + 2) * sizeof(T));
        }
        a.st[s].rp = (int)o;
        o = up16(o + (size_t)a.st[s].bw * a.st[s].bh * sizeof(T));
    }
    // (the planes above are zeroed; everything below is written before it is read)
    a.sm_idle = (int)o; o += 6 * 128;
    a.sm_p = (int)o;
    if (la == 0) o = up16(o + sizeof(T) * B * B * (size_t)nt);
    for (int s = 0; s < ns; ++s) {
        for (int k = 0; k < a.st[s].nlev; ++k) {
            a.st[s].simg[k] = (int)o;
            if (s > 0 || sizeof(T) == 4) o = up16(o + sizeof(T) * table[s][k].size());
        }
        if (s == 0) continue;
        a.st[s].sfm = (int)o;
        o = up16(o + sizeof(int) * (size_t)a.st[s].ni);
        a.st[s].fo = (int)o;
        if (a.st[s].wide) o = up16(o + sizeof(T) * (size_t)a.st[s].ni);
    }
    a.sm_st = (int)o; o = up16(o + sizeof(a.st));
    a.sm_lut = (int)o; o = up16(o + 32 * sizeof(T));
    a.sm_red = (int)o; o = up16(o + 32 * 8);
    a.sm_slot = (int)o; o = up16(o + 2 * CL_MAXC * 8);
    a.sm_xs = (int)o;
    if (la == 0 && sizeof(T) == 4) {
        const int nb = cdiv(L.nx, 64) * cdiv(L.ny, 32);
        o = up16(o + (size_t)cdiv(nb, C) * 8 * 8);
    }
    P->smem = o;
    P->threads = nt;
    if (o > 226 * 1024) return fail();
    int resident = 0;
    if (dispatch<T>(*P, SolveArgs{}, 1, alloc.st, true, &resident) != cudaSuccess || resident < 1) {
        cudaGetLastError();
        return fail();
    }
    // ---- one upload
    std::vector<unsigned char> blob;
    std::vector<std::pair<const void **, size_t>> at;        // pointers and their places in it
    auto put = [&](const void **dst, const void *src, size_t bytes) {
        at.emplace_back(dst, blob.size());
        blob.resize(up16(blob.size() + bytes));
        if (bytes) std::memcpy(&blob[at.back().second], src, bytes);
    };
    put((const void **)&a.rec, rec.data(), rec.size() * sizeof(int4));
    for (int s = 0; s < ns; ++s) {
        ClStageArgs &st = a.st[s];
        for (int k = 0; k < st.nlev; ++k) {
            if (st.l0 + k == 0) continue;
            if (s == 0) put((const void **)&st.kind[k], kind[k].data(), kind[k].size() * sizeof(int));
            put(&st.img[k], table[s][k].data(), table[s][k].size() * sizeof(T));
        }
        put((const void **)&st.fm, fm[s].data(), fm[s].size() * sizeof(int));
    }
    const unsigned char *dev = (const unsigned char *)alloc(blob.data(), blob.size());
    if (!dev) return fail();
    for (const auto &q : at) *q.first = dev + q.second;
    for (int s = 0; s < ns; ++s)
        for (int k = 0; k < a.st[s].nlev; ++k) {
            const ClStageArgs &st = a.st[s];
            const int b = st.B >> k, lev = st.l0 + k;
            if (lev == 0) continue;
            k_cluster_factor<<<4, 256, 0, alloc.st>>>((T *)st.img[k] + (size_t)2 * b * (b + 1) * st.nrec[k], (long long)b * b * st.nrec[k], lev >= ncoarse ? 1 : 0);
            count_launches(1);
        }
    return P;
}

template <class T, int B, bool FIRST, bool MULTI> static cudaError_t launch_k(const ClusterPlan &p, const SolveArgs &sa, int M, cudaStream_t st, bool query, int *active)
{
    auto kern = k_cluster<T, B, FIRST, MULTI, ClLimit<T, B>::threads>;
    if constexpr (sizeof(T) == 8 && B == 2)
        if (p.threads <= CL_FEW_THREADS) kern = k_cluster<T, B, FIRST, MULTI, CL_FEW_BOUND>;
    if constexpr (sizeof(T) == 4 && B == 4 && FIRST)
        if (p.threads <= CL_MID_BOUND && (p.threads > 320 || p.smem > 112 * 1024)) kern = k_cluster<T, B, FIRST, MULTI, CL_MID_BOUND>;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(p.a.C * M);
    cfg.blockDim = dim3(p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.a.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = MULTI ? 1 : 0;
    if (query) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        if (e == cudaSuccess && MULTI) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        if (MULTI) return cudaOccupancyMaxActiveClusters(active, kern, &cfg);
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(active, kern, p.threads, p.smem);
    }
    return cudaLaunchKernelEx(&cfg, kern, p.a, sa);
}
template <class T> static cudaError_t dispatch(const ClusterPlan &p, const SolveArgs &sa, int M, cudaStream_t st, bool query, int *active)
{
    const bool first = p.a.la == 0;
    if constexpr (sizeof(T) == 4) {
        if (!first) return launch_k<T, 4, false, true>(p, sa, M, st, query, active);
        if (p.a.st[0].B == 4 && !p.multi) return launch_k<T, 4, true, false>(p, sa, M, st, query, active);
    }
    if (p.a.st[0].B == 4) return launch_k<T, 4, true, true>(p, sa, M, st, query, active);
    return p.multi ? launch_k<T, 2, true, true>(p, sa, M, st, query, active) : launch_k<T, 2, true, false>(p, sa, M, st, query, active);
}

ClusterPlan *cluster_plan(const ClusterHostLevel *hl, int nlev, int ncoarse, bool mixed, int la, const ClusterAlloc &alloc)
{
    // Candidates in order of preference; the first that fits is taken.  The choice depends on the grid
    // and the precision alone, so a member's arithmetic does not depend on how many run beside it.
    struct Cand { int B, C; };
    std::vector<Cand> cand;
    const ClBlocks b2(hl[la], 2), b4(hl[la], 4);
    if (mixed) {
        if (la == 0) cand.push_back({2, 1});
        // The smallest cluster that holds the grid, rounded up to the largest size of which as many are
        // resident (clusters at 180 KB per block, measured: 2: 76, 3 and 4: 36, 5: 28, 6: 23, 7 to 9: 15,
        // 10: 13, 12: 8, 14 and 16: 7): more SMs per member that no other member could use (256 x 128, 33
        // members: 3 blocks 7.8 ms, 4 blocks 7.4 ms, 5 blocks 7.9 ms).
        for (int C : {1, 2, 4, 3, 5, 6, 9, 8, 7, 10, 12, 14, 16}) cand.push_back({4, C});
    } else if (la == 0) {
        // FP64 issues one warp instruction per scheduler in 64 cycles (0.49 FMA per clock and warp, 1.67 per
        // SM from four warps on, measured): about four warps per block, on up to twelve blocks (256 x 128, 17
        // members: 10 blocks 10.7 ms, 12 blocks 9.9 ms, 14 blocks 16.2 ms: one block per SM; 128 x 64, one
        // member: 53.1, 51.8 and 51.8 ms)
        const int four = std::max(1, cdiv(b2.nact, 128)), want = four > 10 ? 12 : four;
        // up to 256 threads of 2 x 2 cells; beyond, 4 x 4 (three levels stay distributed)
        if (b2.nact <= 2560)
            for (int C = want; C <= CL_MAXC; ++C) cand.push_back({2, C});
        for (int C = want; C <= CL_MAXC; ++C) cand.push_back({4, C});
        for (int C = want; C <= CL_MAXC; ++C) cand.push_back({2, C});
        for (int C = want - 1; C >= 1; --C) cand.push_back({2, C});
    }
    for (const Cand &q : cand) {
        const ClBlocks &bl = q.B == 2 ? b2 : b4;
        ClusterPlan *p = mixed ? make_plan<float>(hl, nlev, ncoarse, la, bl, q.C, alloc) : make_plan<double>(hl, nlev, ncoarse, la, bl, q.C, alloc);
        if (p) return p;
    }
    return nullptr;
}
void cluster_plan_free(ClusterPlan *p) { delete p; }

static void set_sweeps(ClusterPlan *p, const PoissonCfg &pc)
{
    p->a.nu[0][0] = pc.nu_pre; p->a.nu[0][1] = pc.nu_post;
    p->a.nu[1][0] = pc.nu_c ? pc.nu_c : pc.nu_pre;
    p->a.nu[1][1] = pc.nu_c ? pc.nu_c : pc.nu_post;
    p->a.coarse_sweeps = pc.coarse_sweeps;
}

template <class T>
void launch_cluster_solve(const Grid &g, const Level &L0, int M, const PoissonBufs &B, const PoissonCfg &pc, const Partials &pt,
                          MemberCtl *ctl, cudaStream_t st)
{
    ClusterPlan *p = pc.solve;
    set_sweeps(p, pc);
    SolveArgs sa{};
    sa.mode = 0;
    sa.wait_limit = pc.wait_limit;
    sa.max_outer = pc.max_outer; sa.max_inner = pc.max_inner;
    sa.inner_rtol2 = pc.inner_rtol2; sa.rtol_abs = pc.rtol_abs;
    sa.mc = pc.mc;
    sa.cxd = L0.cx; sa.cyd = L0.cy; sa.cxf = L0.cxf; sa.cyf = L0.cyf;
    sa.nx = g.nx; sa.ny = g.ny; sa.fluid = g.fluid;
    sa.bh = B.ms.bh; sa.bl = B.ms.bl; sa.xh = B.ms.xh; sa.xl = B.ms.xl;
    sa.b = B.b; sa.x = B.x; sa.acc = B.e;
    sa.rc = make_ctx(pt);
    sa.ctl = ctl;
    if (pc.conditional_loop) {
        sa.first_o = 0; sa.one = 0; sa.count_last = 1;
        if (dispatch<T>(*p, sa, M, st, false, nullptr) != cudaSuccess) note_capture_failure();
        count_launches(1);
        return;
    }
    for (int o = 0; o <= pc.max_outer; ++o) {                // one launch per refinement
        sa.first_o = o; sa.one = 1; sa.count_last = 0;
        if (dispatch<T>(*p, sa, M, st, false, nullptr) != cudaSuccess) note_capture_failure();
        count_launches(1);
    }
}
template void launch_cluster_solve<float>(const Grid &, const Level &, int, const PoissonBufs &, const PoissonCfg &, const Partials &, MemberCtl *, cudaStream_t);
template void launch_cluster_solve<double>(const Grid &, const Level &, int, const PoissonBufs &, const PoissonCfg &, const Partials &, MemberCtl *, cudaStream_t);

void launch_cluster_vcycle(int M, const float *f, float *e, const PoissonCfg &pc, MemberCtl *ctl, int inner_guard, cudaStream_t st)
{
    ClusterPlan *p = pc.coarse;
    set_sweeps(p, pc);
    SolveArgs sa{};
    sa.mode = 1;
    sa.inner_guard = inner_guard;
    sa.wait_limit = pc.wait_limit;
    sa.f = f; sa.e = e;
    sa.ctl = ctl;
    if (dispatch<float>(*p, sa, M, st, false, nullptr) != cudaSuccess) note_capture_failure();
    count_launches(1);
}

} // namespace envar
