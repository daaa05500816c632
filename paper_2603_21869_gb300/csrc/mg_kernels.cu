// Multigrid kernels for the pressure Poisson equation A p = b, A = -Laplacian
// with one ghost layer (Section 2.4: Eq. neg_lap_discretize, the printed
// 3x3x3 kernel, Eq. jacobi_pc, Eqs. restriction / prolongation, Algorithm 1).
//
// The solve runs in correction form: the level-0 residual r = b - A p is
// formed from the FP64 pressure with an FP64 norm, a V-cycle computes the
// correction e from A e = r in the inner precision (FP64, FP32 or BF16
// storage), and the last post-smoothing sweep adds e to p.  In exact
// arithmetic this is the V-cycle on p itself; in finite precision it is
// defect correction with an FP64 outer residual.
//
//   smoother   e <- e + w_J (r - A e) / D, D = sum_active 2 / h_a^2
//   RES        coarse r = mean of the children's residuals r - A e
//   PROL       e += trilinear interpolation of the coarse correction:
//              3/4 parent + 1/4 neighbour per axis, neighbour index clamped
//   coarsest   e = A^{-1} r with the dense inverse built on the host
//
// Every cell carries a 16-bit neighbour code (two bits per face: 0 = fluid
// neighbour, 1 = zero-gradient ghost, 2 = zero-value ghost; bit 12 = solid),
// so the stencil needs one small load instead of mask and face-table lookups.
// Grid kernels use 3D blocks (no integer division).  The coarse levels are
// cycled by one cluster of blocks (coarse_kernels.cu).  The level-0 residual
// kernel finishes the norm in its last block and decides on the device
// whether another cycle runs, so the whole solve can live in a CUDA graph.
#include "fp_convert.h"
#include "fvm_internal.cuh"

namespace {

template <class T> struct Acc { using type = T; };
template <> struct Acc<__nv_bfloat16> { using type = float; };

constexpr int BX = 32, BY = 4, BZ = 2;

__device__ __forceinline__ bool cell3(const LevelDev& L, const BlockAt& at, int& i, int& j, int& k) {
    i = at.b.x * BX + threadIdx.x;
    j = at.b.y * BY + threadIdx.y;
    k = at.b.z * BZ + threadIdx.z;
    return i < L.n[0] && j < L.n[1] && k < L.n[2];
}

// value across one face: the neighbour (read through `get`, only for code 0),
// the zero-gradient ghost eP or the zero-value ghost -eP
template <class C, class G>
__device__ __forceinline__ C nb_val(uint32_t code, int idx, C eP, G get) {
    return code == 0 ? get(idx) : (code == 1 ? eP : -eP);
}

// (A e)_P = sum_active (2 eP - e_lo - e_hi) / h_a^2; get(q) reads e at cell q
template <class C, class G>
__device__ __forceinline__ C apply_A_with(const LevelDev& L, uint32_t f, int c, C eP, G get) {
    const int sx = 1, sy = L.n[0], sz = L.n[0] * L.n[1];
    C acc = (C)0;
    if (L.active[0]) {
        const C lo = nb_val<C>(f & 3u, c - sx, eP, get), hi = nb_val<C>((f >> 2) & 3u, c + sx, eP, get);
        acc += ((eP - lo) + (eP - hi)) * LP<C>::ih2(L, 0);
    }
    if (L.active[1]) {
        const C lo = nb_val<C>((f >> 4) & 3u, c - sy, eP, get), hi = nb_val<C>((f >> 6) & 3u, c + sy, eP, get);
        acc += ((eP - lo) + (eP - hi)) * LP<C>::ih2(L, 1);
    }
    if (L.active[2]) {
        const C lo = nb_val<C>((f >> 8) & 3u, c - sz, eP, get), hi = nb_val<C>((f >> 10) & 3u, c + sz, eP, get);
        acc += ((eP - lo) + (eP - hi)) * LP<C>::ih2(L, 2);
    }
    return acc;
}

// A e for e in global memory (read-only path)
template <class C, class T>
__device__ __forceinline__ C apply_A(const LevelDev& L, uint32_t f, const T* e, int c, C eP) {
    return apply_A_with<C>(L, f, c, eP, [&](int q) { return to_c<C>(ldg(e + q)); });
}

__device__ __forceinline__ bool is_solid(uint32_t f) { return (f >> 12) & 1u; }

template <class C>
__device__ __forceinline__ C sel(uint32_t code, C nb, C eP) {
    return code == 0 ? nb : (code == 1 ? eP : -eP);
}

// A e at one cell from its gathered neighbours: the general form, with each
// face's ghost chosen by its code.  Kept out of line so that it cannot be
// predicated into the common path below.
template <class C>
__device__ __noinline__ C A7_general(const LevelDev& L, uint32_t f, C eP, C xm, C xp, C ym, C yp, C zm, C zp) {
    C acc = (C)0;
    if (L.active[0]) acc += ((eP - sel(f & 3u, xm, eP)) + (eP - sel((f >> 2) & 3u, xp, eP))) * LP<C>::ih2(L, 0);
    if (L.active[1]) acc += ((eP - sel((f >> 4) & 3u, ym, eP)) + (eP - sel((f >> 6) & 3u, yp, eP))) * LP<C>::ih2(L, 1);
    if (L.active[2]) acc += ((eP - sel((f >> 8) & 3u, zm, eP)) + (eP - sel((f >> 10) & 3u, zp, eP))) * LP<C>::ih2(L, 2);
    return acc;
}

// A e at one cell.  The neighbour values are loaded with indices clamped into
// the grid, so at a zero-gradient domain face the load already returns eP,
// the ghost value.  Every cell without a zero-value face or a solid neighbour
// (code bit 13 clear) therefore takes diag eP - sum_a ih2_a (lo + hi), with
// ih2_a = 0 on a collapsed axis; the rest take the general form.
template <class C>
__device__ __forceinline__ C A7(const LevelDev& L, uint32_t f, C eP, C xm, C xp, C ym, C yp, C zm, C zp) {
    if (!((f >> 13) & 1u)) {
        C s = (xm + xp) * LP<C>::ih2a(L, 0);
        s = fma(ym + yp, LP<C>::ih2a(L, 1), s);
        s = fma(zm + zp, LP<C>::ih2a(L, 2), s);
        return fma(LP<C>::diag(L), eP, -s);
    }
    return A7_general<C>(L, f, eP, xm, xp, ym, yp, zm, zp);
}

// ------------------------------------------------------------------ level 0 residual
// The last block of a level-0 residual pass: a fixed-order reduction over
// all blocks' partials (r^2, b^2): thread t sums blocks t, t + NT, ... in
// order (L2 loads, independent), then a fixed shuffle tree and a fixed sum
// over warps, so the result is deterministic; then the stopping rule.
// Returns the decision in thread 0, -1 elsewhere.  Out of line: it runs once
// per launch and would otherwise hold registers in every block.
template <int NT>
__device__ __noinline__ int resid0_finish(const double* partials, int nblk, SolveState* st,
                                          double (*red)[NT / 32]) {
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    double a0 = 0.0, a1 = 0.0;
    for (int x = tid; x < nblk; x += NT) {
        const double2 v = __ldcg((const double2*)partials + x);
        a0 += v.x;
        a1 += v.y;
    }
    for (int off = 16; off > 0; off >>= 1) {
        a0 += __shfl_xor_sync(0xffffffffu, a0, off);
        a1 += __shfl_xor_sync(0xffffffffu, a1, off);
    }
    __syncthreads();
    if ((tid & 31) == 0) {
        red[0][tid >> 5] = a0;
        red[1][tid >> 5] = a1;
    }
    __syncthreads();
    if (tid != 0) return -1;
    a0 = 0.0;
    a1 = 0.0;
    for (int w = 0; w < NT / 32; ++w) {
        a0 += red[0][w];
        a1 += red[1][w];
    }
    st->counter = 0u;
    st->r2 = a0;
    st->b2 = a1;
    const bool finite = isfinite(a0) && isfinite(a1);
    const double rel = a1 > 0.0 ? sqrt(a0 / a1) : 0.0;
    st->rel = finite ? rel : __longlong_as_double(0x7ff8000000000000ll);
    if (!finite) st->nonfinite = 1;
    int go;
    if (st->fixed > 0) go = st->cycles < st->fixed;
    else go = finite && rel > st->tol && st->cycles < st->max_cycles;
    st->active = go;
    if (!go && st->fixed == 0 && finite && rel > st->tol) st->notconv = 1;
    if (go) {
        st->cycles += st->inner;
        st->total_cycles += st->inner;
    }
    return go;
}

// r = b - A p (FP64), first pre-sweep e = w_J r / D, r^2 and b^2 per block;
// the last block sums the partials in a fixed order and applies the stopping rule.
// run() returns the decision (0 / 1) in the thread that made it, else -1.
template <class TB, class TI>
struct Resid0K {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr int kMinBlocks = 4;   // at most 64 registers (the batched form needs them)
    LevelDev L;
    const double* p;
    const TB* b;
    TI* r;
    TI* e;
    double* partials;
    SolveState* st;
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ int run(const BlockAt& at) const;
};

template <class TB, class TI>
__device__ int Resid0K<TB, TI>::run(const BlockAt& at) const {
    using C = typename Acc<TI>::type;
    __shared__ double red[2][BX * BY * BZ / 32];
    __shared__ bool last;
    int i, j, k;
    C r2 = (C)0, b2 = (C)0;     // squares and warp sums in the inner precision, block sums in FP64
    if (cell3(L, at, i, j, k)) {
        const int c = i + L.n[0] * (j + L.n[1] * k);
        const uint32_t f = L.nbf[c];
        // neighbour loads first (clamped indices), then the FP64 stencil
        const int sy = L.n[0], sz = L.n[0] * L.n[1];
        // (reduced-precision cases: p as double-float pairs, summed in FP64 on this small-grid path)
        auto P = [&](int q) { return sizeof(TB) == 8 ? __ldg(p + q) : pp_get(p, q); };
        const double pP = P(c);
        const double xm = P(c - (i > 0 ? 1 : 0)), xp = P(c + (i < L.n[0] - 1 ? 1 : 0));
        const double ym = P(c - (j > 0 ? sy : 0)), yp = P(c + (j < L.n[1] - 1 ? sy : 0));
        const double zm = P(c - (k > 0 ? sz : 0)), zp = P(c + (k < L.n[2] - 1 ? sz : 0));
        const TB braw = ldg(b + c);
        C rc = (C)0, bc = (C)0;
        if (!is_solid(f)) {
            const double bv = to_c<double>(braw);
            const double Ap = A7<double>(L, f, pP, xm, xp, ym, yp, zm, zp);
            const TI rs = from_c<TI, double>(bv - Ap);
            r[c] = rs;
            rc = to_c<C>(rs);
            bc = to_c<C>(braw);
            e[c] = from_c<TI, C>(LP<C>::wJ(L) * rc * LP<C>::iD(L));
        } else {
            r[c] = from_c<TI, C>((C)0);
            e[c] = from_c<TI, C>((C)0);
        }
        r2 = rc * rc;
        b2 = bc * bc;
    }
    const int tid = threadIdx.x + BX * (threadIdx.y + BY * threadIdx.z);
    for (int off = 16; off > 0; off >>= 1) {
        r2 += __shfl_xor_sync(0xffffffffu, r2, off);
        b2 += __shfl_xor_sync(0xffffffffu, b2, off);
    }
    if ((tid & 31) == 0) {
        red[0][tid >> 5] = (double)r2;
        red[1][tid >> 5] = (double)b2;
    }
    __syncthreads();
    const int nblk = at.g.x * at.g.y * at.g.z;
    const int bid = at.b.x + at.g.x * (at.b.y + at.g.y * at.b.z);
    if (tid == 0) {
        double s0 = 0.0, s1 = 0.0;
        for (int w = 0; w < BX * BY * BZ / 32; ++w) {
            s0 += red[0][w];
            s1 += red[1][w];
        }
        partials[2 * bid] = s0;
        partials[2 * bid + 1] = s1;
        __threadfence();
        const unsigned done = atomicAdd(&st->counter, 1u);
        last = done == (unsigned)nblk - 1u;
    }
    __syncthreads();
    if (!last) return -1;
    __threadfence();
    return resid0_finish<BX * BY * BZ>(partials, nblk, st, red);
}

struct SolveBeginK {
    static constexpr int kThreads = 1;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    SolveState* st;
    __device__ bool live() const { return true; }
    __device__ void run(const BlockAt&) const {
        st->cycles = 0;
        st->counter = 0u;
        st->g_counter = 0u;
        st->g_valid = 0;
        st->active = 1;
    }
};

// ------------------------------------------------------------------ grid kernels (one level)
template <class TI>
struct SweepFirstK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev L;
    const TI* r;
    TI* e;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ void run(const BlockAt& at) const {
        using C = typename Acc<TI>::type;
        int i, j, k;
        if (!cell3(L, at, i, j, k)) return;
        const int c = i + L.n[0] * (j + L.n[1] * k);
        const uint32_t f = L.nbf[c];
        e[c] = from_c<TI, C>(is_solid(f) ? (C)0 : LP<C>::wJ(L) * to_c<C>(ldg(r + c)) * LP<C>::iD(L));
    }
};

// store a restricted residual and, where asked (ec0 not null), the coarse
// level's first Jacobi sweep from e = 0 computed from the stored value, as
// SweepFirstK would: one launch fewer per level and V-cycle
template <class TI, class C>
__device__ __forceinline__ void store_restricted(const LevelDev& Lc, TI* rc, TI* ec0, int idx, C val) {
    const TI rs = from_c<TI, C>(val);
    rc[idx] = rs;
    if (ec0)
        ec0[idx] = from_c<TI, C>(is_solid(Lc.nbf[idx]) ? (C)0 : LP<C>::wJ(Lc) * to_c<C>(rs) * LP<C>::iD(Lc));
}

// coarse r = mean over the children of (r - A e); one thread per coarse cell
template <class TI>
struct ResidRestrictK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev Lf, Lc;
    const TI* e;
    const TI* r;
    TI* rc;
    TI* ec0;   // the coarse level's first sweep, or null
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ void run(const BlockAt& at) const;
};

template <class TI>
__device__ void ResidRestrictK<TI>::run(const BlockAt& at) const {
    using C = typename Acc<TI>::type;
    int I, J, K;
    if (!cell3(Lc, at, I, J, K)) return;
    const int fx = Lf.active[0] ? 2 : 1, fy = Lf.active[1] ? 2 : 1, fz = Lf.active[2] ? 2 : 1;
    C sum = (C)0;
    for (int dz = 0; dz < fz; ++dz)
        for (int dy = 0; dy < fy; ++dy)
            for (int dx = 0; dx < fx; ++dx) {
                const int c = (I * fx + dx) + Lf.n[0] * ((J * fy + dy) + Lf.n[1] * (K * fz + dz));
                const uint32_t f = Lf.nbf[c];
                if (is_solid(f)) continue;
                const C eP = to_c<C>(ldg(e + c));
                sum += to_c<C>(ldg(r + c)) - apply_A<C>(Lf, f, e, c, eP);
            }
    store_restricted<TI, C>(Lc, rc, ec0, I + Lc.n[0] * (J + Lc.n[1] * K), sum / (C)(fx * fy * fz));
}

template <class TI>
struct ProlongK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev Lf, Lc;
    const TI* ec;
    TI* e;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ void run(const BlockAt& at) const {
        using C = typename Acc<TI>::type;
        int i, j, k;
        if (!cell3(Lf, at, i, j, k)) return;
        const int c = i + Lf.n[0] * (j + Lf.n[1] * k);
        if (is_solid(Lf.nbf[c])) return;
        const C add = prolong_at<C>(Lf.active, Lc.n, i, j, k, [&](int q) { return to_c<C>(ldg(ec + q)); },
                                    [&](int q) { return (uint32_t)__ldg(Lc.nbf + q); });
        e[c] = from_c<TI, C>(to_c<C>(e[c]) + add);
    }
};

// ------------------------------------------------------------------ marching kernels (levels >= 0)
// Blocks of TX x TY threads over x-y tiles, marching along z.  Neighbour
// loads use indices clamped into the grid (a face outside the domain reads
// the cell itself), so only cells with code bit 13 need the ghost selects.
constexpr int TX = 32, TY = 8;

struct Walk {
    int i, j, k0, sy, sz, im, ip, jm, jp;
};

__device__ __forceinline__ bool walk_setup(const LevelDev& L, const BlockAt& at, int kz, Walk& w) {
    w.i = at.b.x * TX + threadIdx.x;
    w.j = at.b.y * TY + threadIdx.y;
    w.k0 = at.b.z * kz;
    if (w.i >= L.n[0] || w.j >= L.n[1]) return false;
    w.sy = L.n[0];
    w.sz = L.n[0] * L.n[1];
    w.im = w.i > 0 ? -1 : 0;
    w.ip = w.i < L.n[0] - 1 ? 1 : 0;
    w.jm = w.j > 0 ? -w.sy : 0;
    w.jp = w.j < L.n[1] - 1 ? w.sy : 0;
    return true;
}

// Scalar sweep (FP32 and BF16 levels under 2^20 cells of a case alone or with an x extent that is
// not a multiple of 4, FP64 levels with a collapsed x axis): each thread walks KZ cells along z, keeping the z neighbours in
// registers; all loads of its cells are issued before any arithmetic.
// MODE 0: eout = sweep(ein); MODE 1: p += sweep(ein) (last level-0 sweep); MODE 2: the
// result in FP32 (the last level-0 sweep under the flexible-CG acceleration of BF16 levels).
template <class TI, int MODE, int KZ>
struct SweepK {
    static constexpr int kThreads = TX * TY;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev L;
    const TI* ein;
    const TI* r;
    TI* eout;
    double* p;
    const SolveState* st;
    float* z32;   // MODE 2: the result in FP32
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ void run(const BlockAt& at) const;
};

template <class TI, int MODE, int KZ>
__device__ void SweepK<TI, MODE, KZ>::run(const BlockAt& at) const {
    using C = typename Acc<TI>::type;
    Walk w;
    if (!walk_setup(L, at, KZ, w)) return;
    const int nz = L.n[2];
    const int c0 = w.i + w.sy * w.j + w.sz * w.k0;
    const int kn = nz - w.k0 < KZ ? nz - w.k0 : KZ;   // cells of this thread
    C col[KZ + 2], xm[KZ], xp[KZ], ym[KZ], yp[KZ], rr[KZ];
    uint32_t f[KZ];
    col[0] = to_c<C>(ldg(ein + c0 - (w.k0 > 0 ? w.sz : 0)));
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
        if (kk < kn) {
            const int c = c0 + kk * w.sz;
            col[kk + 1] = to_c<C>(ldg(ein + c));
            xm[kk] = to_c<C>(ldg(ein + c + w.im));
            xp[kk] = to_c<C>(ldg(ein + c + w.ip));
            ym[kk] = to_c<C>(ldg(ein + c + w.jm));
            yp[kk] = to_c<C>(ldg(ein + c + w.jp));
            rr[kk] = to_c<C>(ldg(r + c));
            f[kk] = L.nbf[c];
            if (kk == kn - 1)   // the plane above the thread's last cell (itself at the top face)
                col[kk + 2] = w.k0 + kk < nz - 1 ? to_c<C>(ldg(ein + c + w.sz)) : col[kk + 1];
        }
    }
    const C wJ = LP<C>::wJ(L), iD = LP<C>::iD(L);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
        if (kk < kn) {
            const int c = c0 + kk * w.sz;
            const C eP = col[kk + 1];
            const bool solid = is_solid(f[kk]);
            const C v = solid ? (C)0
                              : eP + wJ * (rr[kk] - A7<C>(L, f[kk], eP, xm[kk], xp[kk], ym[kk], yp[kk], col[kk],
                                                          col[kk + 2])) * iD;
            if (MODE == 0) eout[c] = from_c<TI, C>(v);
            else if (MODE == 2) z32[c] = (float)v;
            else if (!solid) {
                if constexpr (sizeof(TI) == 8) p[c] += (double)v;
                else pp_add(p, c, (float)v);
            }
        }
    }
}

// W consecutive x cells per thread (the vector kernels): W = 2 with 128-bit
// loads for FP64 levels, W = 4 for FP32 levels, W = 8 with 128-bit loads for BF16 levels (W = 4,
// 64-bit loads, where nx is not a multiple of 8).  A warp covers W * 32
// cells of a row (or 2, 4, 8 rows of W * 16, W * 8, W * 4 cells: the widest
// segment that divides nx) and marches zc planes in z: rows j +- 1 and the
// plane after next are loaded whole (indices clamped into the grid, so a
// zero-gradient domain face reads the cell itself), the x neighbours come
// from the adjacent lanes by shuffles (the segment's two end cells from
// single loads), and the z neighbours rotate in registers.
__device__ __forceinline__ void bf2_unpack(uint32_t w, float& a, float& b) {
    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
    a = f.x;
    b = f.y;
}
__device__ __forceinline__ uint32_t bf2_pack(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}

template <class TI, int W> struct VecW;
template <> struct VecW<float, 4> {
    static __device__ __forceinline__ void load(const float* p, int c, float (&o)[4]) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p + c));
        o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    }
    static __device__ __forceinline__ void load_rw(const float* p, int c, float (&o)[4]) {
        const float4 v = *reinterpret_cast<const float4*>(p + c);
        o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    }
    static __device__ __forceinline__ void store(float* p, int c, const float (&v)[4]) {
        *reinterpret_cast<float4*>(p + c) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <> struct VecW<float, 8> {
    static __device__ __forceinline__ void store(float* p, int c, const float (&v)[8]) {
        *reinterpret_cast<float4*>(p + c) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(p + c + 4) = make_float4(v[4], v[5], v[6], v[7]);
    }
};
template <> struct VecW<__nv_bfloat16, 4> {
    static __device__ __forceinline__ void load(const __nv_bfloat16* p, int c, float (&o)[4]) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(p + c));
        bf2_unpack(v.x, o[0], o[1]);
        bf2_unpack(v.y, o[2], o[3]);
    }
    static __device__ __forceinline__ void load_rw(const __nv_bfloat16* p, int c, float (&o)[4]) {
        const uint2 v = *reinterpret_cast<const uint2*>(p + c);
        bf2_unpack(v.x, o[0], o[1]);
        bf2_unpack(v.y, o[2], o[3]);
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, int c, const float (&v)[4]) {
        *reinterpret_cast<uint2*>(p + c) = make_uint2(bf2_pack(v[0], v[1]), bf2_pack(v[2], v[3]));
    }
};
template <> struct VecW<__nv_bfloat16, 8> {
    static __device__ __forceinline__ void load(const __nv_bfloat16* p, int c, float (&o)[8]) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(p + c));
        bf2_unpack(v.x, o[0], o[1]);
        bf2_unpack(v.y, o[2], o[3]);
        bf2_unpack(v.z, o[4], o[5]);
        bf2_unpack(v.w, o[6], o[7]);
    }
    static __device__ __forceinline__ void load_rw(const __nv_bfloat16* p, int c, float (&o)[8]) {
        const uint4 v = *reinterpret_cast<const uint4*>(p + c);
        bf2_unpack(v.x, o[0], o[1]);
        bf2_unpack(v.y, o[2], o[3]);
        bf2_unpack(v.z, o[4], o[5]);
        bf2_unpack(v.w, o[6], o[7]);
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, int c, const float (&v)[8]) {
        *reinterpret_cast<uint4*>(p + c) =
            make_uint4(bf2_pack(v[0], v[1]), bf2_pack(v[2], v[3]), bf2_pack(v[4], v[5]), bf2_pack(v[6], v[7]));
    }
};
template <> struct VecW<double, 2> {
    static __device__ __forceinline__ void load_rw(const double* p, int c, double (&o)[2]) {
        const double2 v = *reinterpret_cast<const double2*>(p + c);
        o[0] = v.x; o[1] = v.y;
    }
    static __device__ __forceinline__ void load(const double* p, int c, double (&o)[2]) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(p + c));
        o[0] = v.x; o[1] = v.y;
    }
    static __device__ __forceinline__ void store(double* p, int c, const double (&v)[2]) {
        *reinterpret_cast<double2*>(p + c) = make_double2(v[0], v[1]);
    }
};
// the four-cell loads of the other kernels
template <class TI> using Vec4 = VecW<TI, 4>;

// the W cells' 16-bit neighbour codes
template <int W> __device__ __forceinline__ void codes_w(const uint16_t* f, int c, uint32_t (&o)[W]);
template <> __device__ __forceinline__ void codes_w<4>(const uint16_t* f, int c, uint32_t (&o)[4]) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(f + c));
    o[0] = v.x & 0xffffu; o[1] = v.x >> 16; o[2] = v.y & 0xffffu; o[3] = v.y >> 16;
}
template <> __device__ __forceinline__ void codes_w<8>(const uint16_t* f, int c, uint32_t (&o)[8]) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(f + c));
    o[0] = v.x & 0xffffu; o[1] = v.x >> 16; o[2] = v.y & 0xffffu; o[3] = v.y >> 16;
    o[4] = v.z & 0xffffu; o[5] = v.z >> 16; o[6] = v.w & 0xffffu; o[7] = v.w >> 16;
}

// two values side by side (aligned to the pair)
__device__ __forceinline__ void store2(double* p, int c, const double (&v)[2]) {
    *reinterpret_cast<double2*>(p + c) = make_double2(v[0], v[1]);
}
__device__ __forceinline__ void store2(float* p, int c, const float (&v)[2]) {
    *reinterpret_cast<float2*>(p + c) = make_float2(v[0], v[1]);
}
__device__ __forceinline__ void store2(__nv_bfloat16* p, int c, const __nv_bfloat16 (&v)[2]) {
    *reinterpret_cast<__nv_bfloat162*>(p + c) = __halves2bfloat162(v[0], v[1]);
}

template <> __device__ __forceinline__ void codes_w<1>(const uint16_t* f, int c, uint32_t (&o)[1]) {
    o[0] = __ldg(f + c);
}
template <> __device__ __forceinline__ void codes_w<2>(const uint16_t* f, int c, uint32_t (&o)[2]) {
    const uint32_t v = __ldg(reinterpret_cast<const unsigned int*>(f + c));
    o[0] = v & 0xffffu; o[1] = v >> 16;
}

// The flags of a thread's W cells (4 or 8) from cell c on (LevelDev::grp): whether their codes are
// needed, and whether the x ghosts at the two ends are negated.  An eighth of a byte a cell where
// the codes take two: they are a quarter to a third of the bytes of a BF16 sweep, transfer or
// prolongation, and a row's end at an outlet no longer sends its warp through the general stencil.
struct GroupFlags {
    bool codes, neg_l, neg_r;
};
template <int W> __device__ __forceinline__ GroupFlags group_flags(const uint8_t* grp, int c) {
    const uint32_t b = __ldg(grp + (c >> 3));
    if constexpr (W == 8) return {(b & 0x11u) != 0u, (b & 0x02u) != 0u, (b & 0x40u) != 0u};
    const uint32_t n = b >> (c & 4);
    return {(n & 1u) != 0u, (n & 2u) != 0u, (n & 4u) != 0u};
}
// The kernels with more loads in flight per thread (residual, residual and restriction, inner
// products) have two forms: by the flags, for levels without solid cells, and by the codes.  A
// second, dependent load for some groups of most warps costs a room more than the bytes: 512 x 256
// x 128 cells, BF16: residual 104 us with the codes, 109 with the flags; residual and restriction 42
// and 45; inner products and update 141 and 144 (512 x 128 x 128 FP32 channel: 66 and 59, 30 and
// 25.5, 80 and 67 us, the other way round).  The two round a cell at a zero-value x face differently,
// so a batch with both kinds of level takes the third form, which chooses by the level: a case's
// results do not depend on the other cases (inner products of eight served cases 53 us, by the
// codes throughout 46).
enum { kCodes = 0, kFlags = 1, kByLevel = 2 };
template <int F> __device__ __forceinline__ bool takes_flags(const LevelDev& L) {
    return F == kFlags || (F == kByLevel && !L.solids);
}
// go(form) with the form as a compile-time constant
template <class Go>
static cudaError_t by_form(const LevelDev& L, Go go) {
    const bool solids = g_rec ? (g_rec->solids >> L.level) & 1u : L.solids != 0;
    const bool clear = g_rec ? (g_rec->clear >> L.level) & 1u : L.solids == 0;
    if (solids && clear) return go(std::integral_constant<int, kByLevel>());
    if (solids) return go(std::integral_constant<int, kCodes>());
    return go(std::integral_constant<int, kFlags>());
}

// cells per thread of the vector kernels on a level of this storage type
template <class TI> __device__ __host__ constexpr int vec_w() { return sizeof(TI) == 2 ? 8 : (sizeof(TI) == 4 ? 4 : 2); }

// The register image of W cells as loaded (16 bytes for W = 4 FP32 and W = 8
// BF16), converted to FP32 one value at a time where used: keeps the vector
// kernels' rotating planes at 4 registers each.  A BF16 value is the high half
// of its FP32 pattern, so the conversion is one shift or mask.
template <class TI, int W> struct RawW;
template <> struct RawW<float, 4> {
    using T = float4;
    static __device__ __forceinline__ T load(const float* p, int c) { return __ldg(reinterpret_cast<const float4*>(p + c)); }
    static __device__ __forceinline__ float get(const T& v, int t) {
        return t == 0 ? v.x : (t == 1 ? v.y : (t == 2 ? v.z : v.w));
    }
};
template <> struct RawW<float, 2> {
    using T = float2;
    static __device__ __forceinline__ T load(const float* p, int c) { return __ldg(reinterpret_cast<const float2*>(p + c)); }
    static __device__ __forceinline__ float get(const T& v, int t) { return t == 0 ? v.x : v.y; }
};
template <> struct RawW<__nv_bfloat16, 2> {
    using T = uint32_t;
    static __device__ __forceinline__ T load(const __nv_bfloat16* p, int c) {
        return __ldg(reinterpret_cast<const unsigned int*>(p + c));
    }
    static __device__ __forceinline__ float get(const T& v, int t) {
        return __uint_as_float((t & 1) ? (v & 0xffff0000u) : (v << 16));
    }
};
template <> struct RawW<__nv_bfloat16, 4> {
    using T = uint2;
    static __device__ __forceinline__ T load(const __nv_bfloat16* p, int c) {
        return __ldg(reinterpret_cast<const uint2*>(p + c));
    }
    static __device__ __forceinline__ float get(const T& v, int t) {
        const uint32_t w = (t >> 1) == 0 ? v.x : v.y;
        return __uint_as_float((t & 1) ? (w & 0xffff0000u) : (w << 16));
    }
};
template <> struct RawW<__nv_bfloat16, 8> {
    using T = uint4;
    static __device__ __forceinline__ T load(const __nv_bfloat16* p, int c) {
        return __ldg(reinterpret_cast<const uint4*>(p + c));
    }
    static __device__ __forceinline__ float get(const T& v, int t) {
        const uint32_t w = (t >> 1) == 0 ? v.x : ((t >> 1) == 1 ? v.y : ((t >> 1) == 2 ? v.z : v.w));
        return __uint_as_float((t & 1) ? (w & 0xffff0000u) : (w << 16));
    }
};

template <> struct RawW<double, 2> {
    using T = double2;
    static __device__ __forceinline__ T load(const double* p, int c) { return __ldg(reinterpret_cast<const double2*>(p + c)); }
    static __device__ __forceinline__ double get(const T& v, int t) { return t == 0 ? v.x : v.y; }
};
template <> struct RawW<double, 1> {
    using T = double;
    static __device__ __forceinline__ T load(const double* p, int c) { return __ldg(p + c); }
    static __device__ __forceinline__ double get(const T& v, int) { return v; }
};

// FP64 levels (two cells per thread) are bound by the FP64 pipe, two lanes a clock and SM: ghosts
// are chosen by integer operations (a negation that no instruction takes as a modifier, like a
// second pass over a warp with one irregular cell, costs FP64 instructions), and the stencil takes
// 8 operations a cell, r - A e summed from r on: fma(-diag, e_P, r + sum_a ih_a (lo + hi)).
// Measured against one cell per thread at 256 x 64 x 64 cells: sweep 38.5 -> 23.1 us, residual 70 ->
// 38.8, residual and restriction 38.9 -> 26.9, prolongation 61.5 -> 43.0; the sweep's 8 operations
// are 13.3 us at the pipe's rate.
__device__ __forceinline__ double flipped(double x, bool neg) {
    return __hiloint2double(__double2hiint(x) ^ (int)((unsigned)neg << 31), __double2loint(x));
}
__device__ __forceinline__ double ghost64(uint32_t code, double nb, double eP) {   // (code: the face's two bits)
    return code == 0u ? nb : flipped(eP, code == 2u);
}
// r - A e at one cell, every neighbour as loaded at clamped indices
__device__ __forceinline__ double resid64(uint32_t f, double r, double eP, double xm, double xp, double ym, double yp,
                                          double zm, double zp, double ihx, double ihy, double ihz, double dg) {
    if (f & 0x2000u) {
        xm = ghost64(f & 3u, xm, eP);
        xp = ghost64((f >> 2) & 3u, xp, eP);
        ym = ghost64((f >> 4) & 3u, ym, eP);
        yp = ghost64((f >> 6) & 3u, yp, eP);
        zm = ghost64((f >> 8) & 3u, zm, eP);
        zp = ghost64((f >> 10) & 3u, zp, eP);
    }
    double s = fma(xm + xp, ihx, r);
    s = fma(ym + yp, ihy, s);
    s = fma(zm + zp, ihz, s);
    return fma(-dg, eP, s);
}

// Ask L2 for the line holding p (no register is tied up while it lands): the z-march kernels
// name their rows of the plane three ahead, so that those loads later hit L2 instead of
// waiting out a DRAM round trip.
__device__ __forceinline__ void l2_prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void l1_prefetch(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

template <class TI, int MODE, int W>
struct SweepVK {
    static constexpr int kThreads = TX * TY;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    // at most 64 registers, four blocks per SM (batched too: the few spilled bytes cost less than a
    // block per SM); the eight-cell update of p (MODE 1) at most 80, three blocks.  (Issuing the
    // next plane's loads before the current plane's arithmetic, at 80 / 128 registers, measured
    // slower on the room.)
    static constexpr int kMinBlocks = (W == 8 && MODE == 1) ? 3 : 4;
    LevelDev L;
    const TI* ein;
    const TI* r;
    TI* eout;
    double* p;
    const SolveState* st;
    int zc;    // planes per block
    float* z32;   // MODE 2: the sweep's result in FP32 (the flexible-CG direction of BF16 levels)
    int lrl;   // log2 of the lanes per row segment (5: a warp per W * 32-cell segment; 4, 3, 2: a warp
               // covers 2, 4 or 8 rows, so narrow rows leave no lane idle)
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ void run(const BlockAt& at) const;
};

template <class TI, int MODE, int W>
__device__ void SweepVK<TI, MODE, W>::run(const BlockAt& at) const {
    using C = typename Acc<TI>::type;
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const int LR = 1 << lrl, lane = threadIdx.x & (LR - 1), sub = threadIdx.x >> lrl;
    const int i4 = at.b.x * (W * LR) + lane * W, j = ((at.b.y * TY + threadIdx.y) << (5 - lrl)) + sub;
    const int k0 = at.b.z * zc, k1 = min(nz, k0 + zc);
    const bool in = i4 < nx && j < ny;
    const int sy = nx, sz = nx * ny;
    const int ic = min(i4, nx - W), jc = min(j, ny - 1);
    const int own = ic + sy * jc, om = ic + sy * max(jc - 1, 0), op = ic + sy * min(jc + 1, ny - 1);
    const int xl = max(ic - 1, 0) + sy * jc, xr = min(ic + W, nx - 1) + sy * jc;
    const bool last = i4 + W >= nx;   // the row's last cell is this thread's: its x+ ghost is itself
    const C ihx = LP<C>::ih2a(L, 0), ihy = LP<C>::ih2a(L, 1), ihz = LP<C>::ih2a(L, 2);
    const C dg = LP<C>::diag(L), wiD = LP<C>::wJ(L) * LP<C>::iD(L);
    // the functor's pointers in registers for the whole march
    const TI* const ein = this->ein;
    const TI* const r = this->r;
    TI* const eout = this->eout;
    double* const p = this->p;
    const uint16_t* const nbf = L.nbf;
    using R = RawW<TI, W>;
    typename R::T em = R::load(ein, max(k0 - 1, 0) * sz + own);
    typename R::T ec = R::load(ein, k0 * sz + own);
    typename R::T ep = R::load(ein, min(k0 + 1, nz - 1) * sz + own);
    for (int k = k0; k < k1; ++k) {
        const int base = k * sz;
        uint32_t fs[W];
        const typename R::T ym = R::load(ein, base + om);
        const typename R::T yp = R::load(ein, base + op);
        const typename R::T rr = R::load(r, base + own);
        GroupFlags gf = {true, false, false};
        if constexpr (sizeof(C) == 8) codes_w<W>(nbf, base + own, fs);
        else gf = group_flags<W>(L.grp, base + own);
        const C xls = lane == 0 ? to_c<C>(ldg(ein + base + xl)) : (C)0;
        const C xrs = lane == LR - 1 ? to_c<C>(ldg(ein + base + xr)) : (C)0;
        const typename R::T en = R::load(ein, min(k + 2, nz - 1) * sz + own);   // plane after next
        if (k + 3 < k1 + 2 && k + 3 < nz) {   // this row of the plane three ahead
            const int fb = (k + 3) * sz + own;
            l2_prefetch(ein + fb);
            l2_prefetch(r + fb);
            if constexpr (sizeof(C) == 8) l2_prefetch(nbf + fb);
        }
        // (no L1 prefetch of the next plane here, unlike the residual and inner-product kernels:
        // with two planes a block the sweep measured 2 % faster without it)
        C left = __shfl_up_sync(0xffffffffu, R::get(ec, W - 1), 1, LR);
        C right = __shfl_down_sync(0xffffffffu, R::get(ec, 0), 1, LR);
        if (lane == 0) left = xls;
        if (lane == LR - 1) right = xrs;
        if (last) right = R::get(ec, W - 1);
        if (gf.neg_l) left = -left;   // (a row's first cell: left is the cell itself)
        if (gf.neg_r) right = -right;
        C v[W];
        if constexpr (sizeof(C) == 8) {
#pragma unroll
            for (int t = 0; t < W; ++t) {
                const C eP = R::get(ec, t);
                const C d = resid64(fs[t], R::get(rr, t), eP, t == 0 ? left : R::get(ec, t - 1),
                                    t == W - 1 ? right : R::get(ec, t + 1), R::get(ym, t), R::get(yp, t), R::get(em, t),
                                    R::get(ep, t), ihx, ihy, ihz, dg);
                v[t] = is_solid(fs[t]) ? (C)0 : fma(wiD, d, eP);
            }
        } else if (!gf.codes) {
            // every cell fluid, each ghost the clamped in-grid load: the plain stencil
#pragma unroll
            for (int t = 0; t < W; ++t) {
                const C eP = R::get(ec, t);
                const C xm = t == 0 ? left : R::get(ec, t - 1), xp = t == W - 1 ? right : R::get(ec, t + 1);
                C s = (xm + xp) * ihx;
                s = fma(R::get(ym, t) + R::get(yp, t), ihy, s);
                s = fma(R::get(em, t) + R::get(ep, t), ihz, s);
                v[t] = fma(wiD, R::get(rr, t) - fma(dg, eP, -s), eP);
            }
        } else {
            codes_w<W>(nbf, base + own, fs);
#pragma unroll
            for (int t = 0; t < W; ++t) {
                const C eP = R::get(ec, t);
                const C xm = t == 0 ? left : R::get(ec, t - 1), xp = t == W - 1 ? right : R::get(ec, t + 1);
                const C zm = R::get(em, t), zp = R::get(ep, t), ya = R::get(ym, t), yb = R::get(yp, t);
                C A;
                if (!((fs[t] >> 13) & 1u)) {
                    C s = (xm + xp) * ihx;
                    s = fma(ya + yb, ihy, s);
                    s = fma(zm + zp, ihz, s);
                    A = fma(dg, eP, -s);
                } else {
                    A = A7_general<C>(L, fs[t], eP, xm, xp, ya, yb, zm, zp);
                }
                v[t] = is_solid(fs[t]) ? (C)0 : fma(wiD, R::get(rr, t) - A, eP);
            }
        }
        if (in) {
            if constexpr (MODE == 0) {
                VecW<TI, W>::store(eout, base + own, v);
            } else if constexpr (MODE == 2) {
                VecW<float, W>::store(z32, base + own, v);
            } else if constexpr (sizeof(C) == 8) {
                double o[W];
                VecW<double, W>::load_rw(p, base + own, o);
#pragma unroll
                for (int t = 0; t < W; ++t) o[t] = o[t] + v[t];   // (0 in solid cells)
                VecW<double, W>::store(p, base + own, o);
            } else {   // p (double-float pairs) += the correction, two cells per 16 bytes
                float4* pp = reinterpret_cast<float4*>(p + base + own);
#pragma unroll
                for (int h = 0; h < W / 2; ++h) {
                    float4 a = pp[h];
                    if (!gf.codes || !is_solid(fs[2 * h])) {
                        const float2 x = pp_plus(make_float2(a.x, a.y), v[2 * h]);
                        a.x = x.x;
                        a.y = x.y;
                    }
                    if (!gf.codes || !is_solid(fs[2 * h + 1])) {
                        const float2 x = pp_plus(make_float2(a.z, a.w), v[2 * h + 1]);
                        a.z = x.x;
                        a.w = x.y;
                    }
                    pp[h] = a;
                }
            }
        }
        em = ec;
        ec = ep;
        ep = en;
    }
}

// The last block of a flexible-CG inner-product pass: sums all blocks'
// partials in a fixed order (thread t: blocks t, t + NT, ...; then a fixed
// shuffle tree and a fixed sum over warps) and sets beta, alpha and the kept
// (d, A d).  Out of line: it runs once per launch and would otherwise hold
// registers in every block.
template <int NT>
__device__ __noinline__ void fcg_finish(const double* partials, int nblk, SolveState* st, bool have,
                                        double (*red)[NT / 32]) {
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int x = tid; x < nblk; x += NT) {
        const double2 u = __ldcg(reinterpret_cast<const double2*>(partials + 4 * x));
        const double2 v = __ldcg(reinterpret_cast<const double2*>(partials + 4 * x + 2));
        a[0] += u.x;
        a[1] += u.y;
        a[2] += v.x;
        a[3] += v.y;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m)
        for (int off = 16; off > 0; off >>= 1) a[m] += __shfl_xor_sync(0xffffffffu, a[m], off);
    __syncthreads();
    if ((tid & 31) == 0)
        for (int m = 0; m < 4; ++m) red[m][tid >> 5] = a[m];
    __syncthreads();
    if (tid == 0) {
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        for (int m = 0; m < 4; ++m)
            for (int w = 0; w < NT / 32; ++w) t[m] += red[m][w];
        double beta = (have && st->g_dq > 0.0) ? t[1] / st->g_dq : 0.0;
        double dq = t[0] - beta * t[1];
        if (!(dq > 0.0)) {   // restart along z alone
            beta = 0.0;
            dq = t[0];
        }
        st->g_beta = beta;
        st->g_alpha = dq > 0.0 ? (t[2] - beta * t[3]) / dq : 0.0;
        st->g_dq = dq;
        st->g_valid = 1;
        st->g_counter = 0u;
    }
}

// the four sums of one block (each thread's in s) into partials; the last
// block to finish completes the pass (fcg_finish)
template <int NT, class T>
__device__ __forceinline__ void fcg_reduce(T (&s)[4], double* partials, SolveState* st, bool have,
                                           const BlockAt& at) {
    __shared__ double red[4][NT / 32];
    __shared__ bool last;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
#pragma unroll
    for (int m = 0; m < 4; ++m)
        for (int off = 16; off > 0; off >>= 1) s[m] += __shfl_xor_sync(0xffffffffu, s[m], off);
    if ((tid & 31) == 0)
        for (int m = 0; m < 4; ++m) red[m][tid >> 5] = (double)s[m];
    __syncthreads();
    const int nblk = at.g.x * at.g.y * at.g.z;
    if (tid == 0) {
        const int bid = at.b.x + at.g.x * (at.b.y + at.g.y * at.b.z);
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        for (int w = 0; w < NT / 32; ++w)
            for (int m = 0; m < 4; ++m) t[m] += red[m][w];
        reinterpret_cast<double2*>(partials + 4 * bid)[0] = make_double2(t[0], t[1]);
        reinterpret_cast<double2*>(partials + 4 * bid)[1] = make_double2(t[2], t[3]);
        __threadfence();
        last = atomicAdd(&st->g_counter, 1u) == (unsigned)nblk - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    fcg_finish<NT>(partials, nblk, st, have, red);
}

// ------------------------------------------------------------------ level 0 residual in float-float
// The reduced-precision cases hold p as double-float pairs (pp_load); on large
// levels and in batches this path evaluates r = b - A p without the FP64 pipe
// (1/64 of the FP32 rate here): the stencil runs in double-float arithmetic (Dekker's error-free sum
// and FMA-based product), about 2^-48 relative accuracy.  As a difference
// form, A p = sum_a ih2_a ((P - g_lo) + (P - g_hi)) with g the neighbour
// (code 0), P (zero-gradient: no term) or -P (zero-value: 2P), which equals
// both branches of A7.
__device__ __forceinline__ void ff_load4(const double* p, int c, FF (&o)[4]) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p + c));
    const float4 b = __ldg(reinterpret_cast<const float4*>(p + c) + 1);
    o[0] = {a.x, a.y};
    o[1] = {a.z, a.w};
    o[2] = {b.x, b.y};
    o[3] = {b.z, b.w};
}

// P - ghost across one face: the neighbour (code 0), none (1) or 2P (2)
__device__ __forceinline__ FF ff_face(uint32_t code, FF P, FF nb) {
    const FF d = ff_add(P, ff_neg(nb));
    if (code == 0u) return d;
    if (code == 1u) return {0.0f, 0.0f};
    return {2.0f * P.h, 2.0f * P.l};
}

// one axis of A p at a regular cell: ih (2P - a - b), the neighbours' sum and
// the difference by error-free sums, the products' low parts by FMA; the
// result is left unnormalised (its low part is small against the high part's
// inputs, which is all the sums below need)
__device__ __forceinline__ FF ff_axis(FF P, FF a, FF b, FF ih) {
    const FF s = ff_two_sum(a.h, b.h);
    const float sl = s.l + (a.l + b.l);
    const FF d = ff_two_sum(2.0f * P.h, -s.h);
    const float dl = d.l + (2.0f * P.l - sl);
    const float p = d.h * ih.h;
    float e = fmaf(d.h, ih.h, -p);
    e = fmaf(d.h, ih.l, e);
    e = fmaf(dl, ih.h, e);
    return {p, e};
}

// b - A p rounded to FP32 at a regular cell (code bit 13 clear: the clamped
// loads are the ghosts), ih2 = 0 on a collapsed axis
__device__ __forceinline__ float ff_resid_regular(float b, FF P, FF xm, FF xp, FF ym, FF yp, FF zm, FF zp, FF ihx,
                                                  FF ihy, FF ihz) {
    const FF ax = ff_axis(P, xm, xp, ihx), ay = ff_axis(P, ym, yp, ihy), az = ff_axis(P, zm, zp, ihz);
    const FF t = ff_two_sum(ax.h, ay.h);
    const FF t2 = ff_two_sum(t.h, az.h);
    const float al = (t.l + t2.l) + (ax.l + ay.l + az.l);
    const FF u = ff_two_sum(b, -t2.h);
    return u.h + (u.l - al);
}

// Two cells' double-float values side by side (cells 2q and 2q + 1 of a thread's four) and
// the arithmetic of ff_axis / ff_resid_regular on both at once with the packed FP32
// instructions (add / mul / fma .f32x2: one instruction for the pair, each lane rounded as the
// scalar instruction rounds it).  A difference a - b is fma(b, -1, a), rounded once like the
// scalar subtraction; a negation is a product by -1 (exact).
struct FF2 {
    float2 h, l;
};
__device__ __forceinline__ float2 p2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p2sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 p2neg(float2 a) { return __fmul2_rn(a, make_float2(-1.0f, -1.0f)); }
__device__ __forceinline__ FF2 ff2_two_sum(float2 a, float2 b) {
    const float2 s = p2add(a, b);
    const float2 bb = p2sub(s, a);
    return {s, p2add(p2sub(a, p2sub(s, bb)), p2sub(b, bb))};
}
__device__ __forceinline__ FF2 ff2_axis(FF2 P, FF2 a, FF2 b, float2 ihh, float2 ihl) {
    const FF2 s = ff2_two_sum(a.h, b.h);
    const float2 sl = p2add(s.l, p2add(a.l, b.l));
    const FF2 d = ff2_two_sum(p2add(P.h, P.h), p2neg(s.h));
    const float2 dl = p2add(d.l, p2sub(p2add(P.l, P.l), sl));
    const float2 p = __fmul2_rn(d.h, ihh);
    float2 e = __ffma2_rn(d.h, ihh, p2neg(p));
    e = __ffma2_rn(d.h, ihl, e);
    e = __ffma2_rn(dl, ihh, e);
    return {p, e};
}
__device__ __forceinline__ float2 ff2_resid_regular(float2 b, FF2 P, FF2 xm, FF2 xp, FF2 ym, FF2 yp, FF2 zm, FF2 zp,
                                                    const float2 ih[6]) {
    const FF2 ax = ff2_axis(P, xm, xp, ih[0], ih[1]), ay = ff2_axis(P, ym, yp, ih[2], ih[3]);
    const FF2 az = ff2_axis(P, zm, zp, ih[4], ih[5]);
    const FF2 t = ff2_two_sum(ax.h, ay.h);
    const FF2 t2 = ff2_two_sum(t.h, az.h);
    const float2 al = p2add(p2add(t.l, t2.l), p2add(p2add(ax.l, ay.l), az.l));
    const FF2 u = ff2_two_sum(b, p2neg(t2.h));
    return p2add(u.h, p2sub(u.l, al));
}
__device__ __forceinline__ FF2 ff2_of(const FF& a, const FF& b) { return {make_float2(a.h, b.h), make_float2(a.l, b.l)}; }

// the same for any cell, each face's ghost chosen by its code (out of line: rare)
__device__ __noinline__ float ff_resid_general(uint32_t f, float b, FF P, FF xm, FF xp, FF ym, FF yp, FF zm, FF zp,
                                               FF ihx, FF ihy, FF ihz) {
    const FF ax = ff_mul(ff_add(ff_face(f & 3u, P, xm), ff_face((f >> 2) & 3u, P, xp)), ihx);
    const FF ay = ff_mul(ff_add(ff_face((f >> 4) & 3u, P, ym), ff_face((f >> 6) & 3u, P, yp)), ihy);
    const FF az = ff_mul(ff_add(ff_face((f >> 8) & 3u, P, zm), ff_face((f >> 10) & 3u, P, zp)), ihz);
    const FF A = ff_add(ff_add(ax, ay), az);
    const FF rr = ff_add(FF{b, 0.0f}, ff_neg(A));
    return rr.h + rr.l;
}

template <class TI> __device__ __forceinline__ float round_inner(float v) { return v; }
template <> __device__ __forceinline__ float round_inner<__nv_bfloat16>(float v) {
    return __bfloat162float(__float2bfloat16_rn(v));
}

// block sums in FP64, then the last block's fixed-order reduction and the stopping rule (the
// decision in the deciding thread, -1 elsewhere)
template <int NT>
__device__ __forceinline__ int resid0_sums(double s0, double s1, double* partials, SolveState* st, const BlockAt& at) {
    __shared__ double red[2][NT / 32];
    __shared__ bool last;
    const int tid = threadIdx.x + TX * threadIdx.y;
    for (int off = 16; off > 0; off >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, off);
        s1 += __shfl_xor_sync(0xffffffffu, s1, off);
    }
    if ((tid & 31) == 0) {
        red[0][tid >> 5] = s0;
        red[1][tid >> 5] = s1;
    }
    __syncthreads();
    const int nblk = at.g.x * at.g.y * at.g.z;
    if (tid == 0) {
        const int bid = at.b.x + at.g.x * (at.b.y + at.g.y * at.b.z);
        double a0 = 0.0, a1 = 0.0;
        for (int w = 0; w < NT / 32; ++w) {
            a0 += red[0][w];
            a1 += red[1][w];
        }
        reinterpret_cast<double2*>(partials)[bid] = make_double2(a0, a1);
        __threadfence();
        last = atomicAdd(&st->counter, 1u) == (unsigned)nblk - 1u;
    }
    __syncthreads();
    if (!last) return -1;
    __threadfence();
    return resid0_finish<NT>(partials, nblk, st, red);
}

// r = b - A p (float-float), r^2 and b^2, the first pre-sweep e = w_J r / D;
// four x cells per thread and a z march (the sweep's layout).  FP32 b, nx % 4 = 0.
template <class TI, int F>   // F: kCodes, kFlags or kByLevel
struct Resid0V4K {
    static constexpr int kThreads = TX * TY;
    static constexpr int kMinBlocks = 3;       // at most 80 registers
    // the batched form needs more (BF16 spills at 80; with FP32 corrections 80 registers, three
    // blocks per SM, measured slower on 64 channels than 128 and two)
    static constexpr int kMinBlocksMany = 2;
    LevelDev L;
    const double* p;
    const float* b;
    TI* r;
    TI* e;
    double* partials;
    SolveState* st;
    int zc;    // planes per block
    int lrl;   // log2 of the lanes per row segment (as in SweepVK)
    __device__ bool live() const { return st->active != 0; }
    __device__ int run(const BlockAt& at) const;
};

template <class TI, int F>
__device__ int Resid0V4K<TI, F>::run(const BlockAt& at) const {
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const int LR = 1 << lrl, lane = threadIdx.x & (LR - 1), sub = threadIdx.x >> lrl;
    const int i4 = at.b.x * (4 * LR) + lane * 4, j = ((at.b.y * TY + threadIdx.y) << (5 - lrl)) + sub;
    const int k0 = at.b.z * zc, k1 = min(nz, k0 + zc);
    const bool in = i4 < nx && j < ny;
    const int sy = nx, sz = nx * ny;
    const int ic = min(i4, nx - 4), jc = min(j, ny - 1);
    const int own = ic + sy * jc, om = ic + sy * max(jc - 1, 0), op = ic + sy * min(jc + 1, ny - 1);
    const int xl = max(ic - 1, 0) + sy * jc, xr = min(ic + 4, nx - 1) + sy * jc;
    const bool lastc = i4 + 4 >= nx;
    const FF ihx = {L.ih2af[0], L.ih2alo[0]}, ihy = {L.ih2af[1], L.ih2alo[1]}, ihz = {L.ih2af[2], L.ih2alo[2]};
    const float2 ih2[6] = {make_float2(ihx.h, ihx.h), make_float2(ihx.l, ihx.l), make_float2(ihy.h, ihy.h),
                           make_float2(ihy.l, ihy.l), make_float2(ihz.h, ihz.h), make_float2(ihz.l, ihz.l)};
    const float wJ = LP<float>::wJ(L), iD = LP<float>::iD(L);
    const double* const pp = this->p;
    const uint16_t* const nbf = L.nbf;
    const bool flags = takes_flags<F>(L);
    FF em[4], ec[4], ep[4];
    ff_load4(pp, max(k0 - 1, 0) * sz + own, em);
    ff_load4(pp, k0 * sz + own, ec);
    ff_load4(pp, min(k0 + 1, nz - 1) * sz + own, ep);
    float r2 = 0.0f, b2 = 0.0f;
    for (int k = k0; k < k1; ++k) {
        const int base = k * sz;
        FF ym[4], yp[4], en[4];
        ff_load4(pp, base + om, ym);
        ff_load4(pp, base + op, yp);
        const float4 bq = __ldg(reinterpret_cast<const float4*>(b + base + own));
        GroupFlags gf = {true, false, false};
        if (flags) gf = group_flags<4>(L.grp, base + own);
        uint32_t fs[4] = {0u, 0u, 0u, 0u};
        if (gf.codes) codes_w<4>(nbf, base + own, fs);
        const FF xls = lane == 0 ? pp_load(pp, base + xl) : FF{0.0f, 0.0f};
        const FF xrs = lane == LR - 1 ? pp_load(pp, base + xr) : FF{0.0f, 0.0f};
        ff_load4(pp, min(k + 2, nz - 1) * sz + own, en);
        if (k + 3 < k1 + 2 && k + 3 < nz) {   // this row of the plane three ahead
            const int fb = (k + 3) * sz + own;
            l2_prefetch(pp + fb);
            l2_prefetch(pp + fb + 2);
            l2_prefetch(b + fb);
            if (!flags) l2_prefetch(nbf + fb);
        }
        if (k + 1 < k1) {   // the next plane's rows into L1 (their loads open the next iteration)
            const int nb = (k + 1) * sz;
            l1_prefetch(pp + nb + om);
            l1_prefetch(pp + nb + op);
            l1_prefetch(b + nb + own);
            if (!flags) l1_prefetch(nbf + nb + own);
        }
        FF left = {__shfl_up_sync(0xffffffffu, ec[3].h, 1, LR), __shfl_up_sync(0xffffffffu, ec[3].l, 1, LR)};
        FF right = {__shfl_down_sync(0xffffffffu, ec[0].h, 1, LR), __shfl_down_sync(0xffffffffu, ec[0].l, 1, LR)};
        if (lane == 0) left = xls;
        if (lane == LR - 1) right = xrs;
        if (lastc) right = ec[3];
        if constexpr (F != kCodes) {   // (at a row's ends left / right is the cell itself)
            if (gf.neg_l) left = ff_neg(left);
            if (gf.neg_r) right = ff_neg(right);
        }
        const FF xs[6] = {left, ec[0], ec[1], ec[2], ec[3], right};
        const float bb[4] = {bq.x, bq.y, bq.z, bq.w};
        // b - A p: a pair of regular cells (code bit 13 clear) in the packed form, any other cell alone
        float rfs[4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int t0 = 2 * q, t1 = t0 + 1;
            if (!(((fs[t0] | fs[t1]) >> 13) & 1u)) {
                const float2 rr = ff2_resid_regular(
                    make_float2(bb[t0], bb[t1]), ff2_of(xs[t0 + 1], xs[t1 + 1]), ff2_of(xs[t0], xs[t1]),
                    ff2_of(xs[t0 + 2], xs[t1 + 2]), ff2_of(ym[t0], ym[t1]), ff2_of(yp[t0], yp[t1]),
                    ff2_of(em[t0], em[t1]), ff2_of(ep[t0], ep[t1]), ih2);
                rfs[t0] = rr.x;
                rfs[t1] = rr.y;
            } else {
#pragma unroll
                for (int t = t0; t <= t1; ++t)
                    rfs[t] = !((fs[t] >> 13) & 1u)
                                 ? ff_resid_regular(bb[t], xs[t + 1], xs[t], xs[t + 2], ym[t], yp[t], em[t], ep[t], ihx,
                                                    ihy, ihz)
                                 : ff_resid_general(fs[t], bb[t], xs[t + 1], xs[t], xs[t + 2], ym[t], yp[t], em[t],
                                                    ep[t], ihx, ihy, ihz);
            }
        }
        float rv[4], ev[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float rf = rfs[t];
            const bool fluid = !is_solid(fs[t]);
            const float rc = fluid ? round_inner<TI>(rf) : 0.0f;
            rv[t] = rc;
            ev[t] = wJ * rc * iD;
            if (in) {
                r2 = fmaf(rc, rc, r2);
                if (fluid) b2 = fmaf(bb[t], bb[t], b2);
            }
        }
        if (in) {
            Vec4<TI>::store(r, base + own, rv);
            Vec4<TI>::store(e, base + own, ev);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            em[t] = ec[t];
            ec[t] = ep[t];
            ep[t] = en[t];
        }
    }
    return resid0_sums<kThreads>((double)r2, (double)b2, partials, st, at);
}

// r = b - A p, r^2 and b^2 and the first pre-sweep in FP64: two x cells per thread and a z march (the
// sweep's layout); a thread's squares are summed in registers, one warp reduction a block (the
// one-cell form's per-cell reduction was 10 of its 24 FP64 operations a cell).  FP64 levels, and the
// FP32 and BF16 cases under 2^20 cells stepped alone: there p's double-float pairs are summed to FP64
// and r is rounded once, as in Resid0K (430,080 cells, us a launch: one cell per thread 47, this with
// conversion instructions 44, with fp_convert.h 32; the double-float form of the large levels 20, with
// errors of the size of p's last bits).
template <class TB, class TI>
struct Resid0DK {
    static constexpr int kThreads = TX * TY;
    static constexpr int kMinBlocks = sizeof(TB) == 8 ? 4 : 3;   // at most 64 registers, 80 with pairs
    LevelDev L;
    const double* p;
    const TB* b;
    TI* r;
    TI* e;
    double* partials;
    SolveState* st;
    int zc;    // planes per block
    int lrl;   // log2 of the lanes per row segment (as in SweepVK)
    __device__ bool live() const { return st->active != 0; }
    __device__ int run(const BlockAt& at) const;
};

template <class TB, class TI>
__device__ int Resid0DK<TB, TI>::run(const BlockAt& at) const {
    using C = typename Acc<TI>::type;
    using R = RawW<double, 2>;   // (a pair has a value's size)
    using RB = RawW<TB, 2>;
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const int LR = 1 << lrl, lane = threadIdx.x & (LR - 1), sub = threadIdx.x >> lrl;
    const int i2 = at.b.x * (2 * LR) + lane * 2, j = ((at.b.y * TY + threadIdx.y) << (5 - lrl)) + sub;
    const int k0 = at.b.z * zc, k1 = min(nz, k0 + zc);
    const bool in = i2 < nx && j < ny;
    const int sy = nx, sz = nx * ny;
    const int ic = min(i2, nx - 2), jc = min(j, ny - 1);
    const int own = ic + sy * jc, om = ic + sy * max(jc - 1, 0), op = ic + sy * min(jc + 1, ny - 1);
    const int xl = max(ic - 1, 0) + sy * jc, xr = min(ic + 2, nx - 1) + sy * jc;
    const double ihx = L.ih2a[0], ihy = L.ih2a[1], ihz = L.ih2a[2], dg = L.diag;
    // values of p as loaded, in FP64: the values themselves, or the sums of their pairs
    auto values = [](const auto& raw, auto& v) {
        constexpr int n = sizeof(v) / sizeof(double);
        if constexpr (sizeof(TB) == 8) {
#pragma unroll
            for (int q = 0; q < n; ++q) v[q] = raw[q];
        } else {
            float x[2 * n];
            double y[2 * n];
#pragma unroll
            for (int q = 0; q < n; ++q) {
                x[2 * q] = __int_as_float(__double2loint(raw[q]));
                x[2 * q + 1] = __int_as_float(__double2hiint(raw[q]));
            }
            widened(x, y);
#pragma unroll
            for (int q = 0; q < n; ++q) v[q] = y[2 * q] + y[2 * q + 1];
        }
    };
    double em[2], ec[2];
    {
        const double2 a = R::load(p, max(k0 - 1, 0) * sz + own), c = R::load(p, k0 * sz + own);
        const double raw[4] = {a.x, a.y, c.x, c.y};
        double v[4];
        values(raw, v);
        em[0] = v[0]; em[1] = v[1];
        ec[0] = v[2]; ec[1] = v[3];
    }
    double r2 = 0.0, b2 = 0.0;
    for (int k = k0; k < k1; ++k) {
        const int base = k * sz;
        const double2 e = R::load(p, min(k + 1, nz - 1) * sz + own), m = R::load(p, base + om), q = R::load(p, base + op);
        const typename RB::T bv = RB::load(b, base + own);
        const double raw[8] = {e.x, e.y, m.x, m.y, q.x, q.y, __ldg(p + base + xl), __ldg(p + base + xr)};
        double v[8];   // k + 1; j - 1; j + 1; left, right
        values(raw, v);
        const TB bt[2] = {RB::get(bv, 0), RB::get(bv, 1)};
        double bd[2];
        widened(bt, bd);
        uint32_t fs[2];
        codes_w<2>(L.nbf, base + own, fs);
        const double rd[2] = {resid64(fs[0], bd[0], ec[0], v[6], ec[1], v[2], v[4], em[0], v[0], ihx, ihy, ihz, dg),
                              resid64(fs[1], bd[1], ec[1], ec[0], v[7], v[3], v[5], em[1], v[1], ihx, ihy, ihz, dg)};
        C rv[2];
        narrowed(rd, rv);   // (BF16: by way of FP32, as from_c does)
        if (in) {
            const TI rs[2] = {from_c<TI, C>(is_solid(fs[0]) ? (C)0 : rv[0]), from_c<TI, C>(is_solid(fs[1]) ? (C)0 : rv[1])};
            const C va = to_c<C>(rs[0]), vc = to_c<C>(rs[1]);
            const C ba = is_solid(fs[0]) ? (C)0 : (C)bt[0], bc = is_solid(fs[1]) ? (C)0 : (C)bt[1];
            const C w = LP<C>::wJ(L), iD = LP<C>::iD(L);
            store2(r, base + own, rs);
            if constexpr (sizeof(TI) == 8) {
                const double wiD = w * iD;
                const TI es[2] = {wiD * va, wiD * vc};
                store2(this->e, base + own, es);
                r2 = fma(va, va, fma(vc, vc, r2));
                b2 = fma(ba, ba, fma(bc, bc, b2));
            } else {   // (squares in FP32 as in Resid0K, the sums in FP64)
                const TI es[2] = {from_c<TI, C>(w * va * iD), from_c<TI, C>(w * vc * iD)};
                store2(this->e, base + own, es);
                const float sq[2] = {fmaf(va, va, vc * vc), fmaf(ba, ba, bc * bc)};
                double sd[2];
                widened(sq, sd);
                r2 += sd[0];
                b2 += sd[1];
            }
        }
        em[0] = ec[0]; em[1] = ec[1];
        ec[0] = v[0]; ec[1] = v[1];
    }
    return resid0_sums<kThreads>(r2, b2, partials, st, at);
}

// The flexible-CG inner products with W x cells per thread and a z march
// (the sweep's layout and neighbour scheme): products, the thread's and the
// warp's sums in T, block and grid sums in FP64.  Needs nx % W = 0.
// (TR: storage of r; TZ: storage of z and the kept direction, FP32 on BF16 levels)
template <class TR, class TZ, int W, int F, class T>   // F: kCodes, kFlags or kByLevel
struct FcgDotVK {
    static constexpr int kThreads = TX * TY;
    static constexpr int kMinBlocks = sizeof(T) > sizeof(TZ) ? 3 : 4;   // at most 64 registers (FP64 sums of FP32 fields: 80)
    static constexpr int kMinBlocksMany = 3;   // the batched form: at most 80 registers
    LevelDev L;
    const TZ* z;
    const TR* r;
    const TZ* dp;
    double* partials;
    SolveState* st;
    int zc;    // planes per block
    int lrl;   // log2 of the lanes per row segment (as in SweepVK)
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const;
};

template <class TR, class TZ, int W, int F, class T>
__device__ void FcgDotVK<TR, TZ, W, F, T>::run(const BlockAt& at) const {
    using C = typename Acc<TZ>::type;
    using R = RawW<TZ, W>;
    using RR = RawW<TR, W>;
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const int LR = 1 << lrl, lane = threadIdx.x & (LR - 1), sub = threadIdx.x >> lrl;
    const int i4 = at.b.x * (W * LR) + lane * W, j = ((at.b.y * TY + threadIdx.y) << (5 - lrl)) + sub;
    const int k0 = at.b.z * zc, k1 = min(nz, k0 + zc);
    const bool in = i4 < nx && j < ny;
    const int sy = nx, sz = nx * ny;
    const int ic = min(i4, nx - W), jc = min(j, ny - 1);
    const int own = ic + sy * jc, om = ic + sy * max(jc - 1, 0), op = ic + sy * min(jc + 1, ny - 1);
    const int xl = max(ic - 1, 0) + sy * jc, xr = min(ic + W, nx - 1) + sy * jc;
    const bool lastc = i4 + W >= nx;
    const C ihx = LP<C>::ih2a(L, 0), ihy = LP<C>::ih2a(L, 1), ihz = LP<C>::ih2a(L, 2);
    const C dg = LP<C>::diag(L);
    const bool have = st->g_valid != 0;
    const TZ* const zz = this->z;
    const uint16_t* const nbf = L.nbf;
    const bool flags = takes_flags<F>(L);
    typename R::T em = R::load(zz, max(k0 - 1, 0) * sz + own);
    typename R::T ec = R::load(zz, k0 * sz + own);
    typename R::T ep = R::load(zz, min(k0 + 1, nz - 1) * sz + own);
    T a0 = (T)0, a1 = (T)0, a2 = (T)0, a3 = (T)0;
    for (int k = k0; k < k1; ++k) {
        const int base = k * sz;
        const typename R::T ym = R::load(zz, base + om);
        const typename R::T yp = R::load(zz, base + op);
        const typename RR::T rr = RR::load(r, base + own);
        typename R::T dd = {};
        if (have) dd = R::load(dp, base + own);
        uint32_t fs[W];
        GroupFlags gf = {true, false, false};
        if (flags) gf = group_flags<W>(L.grp, base + own);
        if (gf.codes) codes_w<W>(nbf, base + own, fs);
        const C xls = lane == 0 ? to_c<C>(ldg(zz + base + xl)) : (C)0;
        const C xrs = lane == LR - 1 ? to_c<C>(ldg(zz + base + xr)) : (C)0;
        const typename R::T en = R::load(zz, min(k + 2, nz - 1) * sz + own);
        if (k + 3 < k1 + 2 && k + 3 < nz) {   // this row of the plane three ahead
            const int fb = (k + 3) * sz + own;
            l2_prefetch(zz + fb);
            l2_prefetch(r + fb);
            if (!flags) l2_prefetch(nbf + fb);
            if (have) l2_prefetch(dp + fb);
        }
        if (k + 1 < k1) {   // the next plane's rows into L1 (their loads open the next iteration)
            const int nb = (k + 1) * sz;
            l1_prefetch(zz + nb + om);
            l1_prefetch(zz + nb + op);
            l1_prefetch(r + nb + own);
            if (!flags) l1_prefetch(nbf + nb + own);
            if (have) l1_prefetch(dp + nb + own);
        }
        C left = __shfl_up_sync(0xffffffffu, R::get(ec, W - 1), 1, LR);
        C right = __shfl_down_sync(0xffffffffu, R::get(ec, 0), 1, LR);
        if (lane == 0) left = xls;
        if (lane == LR - 1) right = xrs;
        if (lastc) right = R::get(ec, W - 1);
        if (flags) {   // (at a row's ends left / right is the cell itself)
            if (gf.neg_l) left = -left;
            if (gf.neg_r) right = -right;
        } else {
            uint32_t any = 0u;   // solid (bit 12) or irregular (bit 13) anywhere among the W cells
#pragma unroll
            for (int t = 0; t < W; ++t) any |= fs[t];
            gf.codes = (any & 0x3000u) != 0u;
        }
        if (in) {
            C zs[W], As[W], ds[W], rs[W];   // (sums in a wider type: the plane's factors, converted together)
#pragma unroll
            for (int t = 0; t < W; ++t) {
                const bool plain = !gf.codes;   // every cell fluid with in-grid ghosts
                if constexpr (sizeof(T) > sizeof(C)) zs[t] = As[t] = ds[t] = rs[t] = (C)0;
                if (!plain && is_solid(fs[t])) continue;
                const C eP = R::get(ec, t);
                const C xm = t == 0 ? left : R::get(ec, t - 1), xp = t == W - 1 ? right : R::get(ec, t + 1);
                const C ya = R::get(ym, t), yb = R::get(yp, t), za = R::get(em, t), zb = R::get(ep, t);
                C A;
                if constexpr (sizeof(C) == 8) {
                    A = -resid64(fs[t], 0.0, eP, xm, xp, ya, yb, za, zb, ihx, ihy, ihz, dg);
                } else if (plain || !((fs[t] >> 13) & 1u)) {
                    C q = (xm + xp) * ihx;
                    q = fma(ya + yb, ihy, q);
                    q = fma(za + zb, ihz, q);
                    A = fma(dg, eP, -q);
                } else {
                    A = A7_general<C>(L, fs[t], eP, xm, xp, ya, yb, za, zb);
                }
                const C d = R::get(dd, t), rv = RR::get(rr, t);
                if constexpr (sizeof(T) > sizeof(C)) {
                    zs[t] = eP;
                    As[t] = A;
                    ds[t] = d;
                    rs[t] = rv;
                } else {
                    a0 = fma(eP, A, a0);
                    a1 = fma(A, d, a1);
                    a2 = fma(rv, eP, a2);
                    a3 = fma(rv, d, a3);
                }
            }
            if constexpr (sizeof(T) > sizeof(C)) {
                T zt[W], At[W], dt[W], rt[W];
                widened(zs, zt);
                widened(As, At);
                widened(ds, dt);
                widened(rs, rt);
#pragma unroll
                for (int t = 0; t < W; ++t) {
                    a0 = fma(zt[t], At[t], a0);
                    a1 = fma(At[t], dt[t], a1);
                    a2 = fma(rt[t], zt[t], a2);
                    a3 = fma(rt[t], dt[t], a3);
                }
            }
        }
        em = ec;
        ec = ep;
        ep = en;
    }
    T s[4] = {a0, a1, a2, a3};
    fcg_reduce<kThreads>(s, partials, st, have, at);
}

// d = z - beta d_prev, p += alpha d (fluid cells), d kept: W consecutive
// cells per thread, one-dimensional grid, d and alpha d in T.  Needs N % W = 0.
template <class TZ, int W, class T>
struct FcgUpdVK {
    static constexpr int kThreads = 256;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev L;
    const TZ* z;
    TZ* dp;
    double* p;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const {
        const int c = W * (at.b.x * kThreads + threadIdx.x);
        if (c >= L.N) return;
        using C = typename Acc<TZ>::type;
        const T alpha = (T)st->g_alpha, beta = (T)st->g_beta;
        C zv[W], dv[W];
#pragma unroll
        for (int t = 0; t < W; ++t) dv[t] = (C)0;
        VecW<TZ, W>::load(z, c, zv);
        if (beta != (T)0) VecW<TZ, W>::load_rw(dp, c, dv);
        uint32_t fs[W];
        GroupFlags gf = {true, false, false};
        if constexpr (sizeof(C) == 4) gf = group_flags<W>(L.grp, c);
        const bool codes = gf.codes;
        if (codes) codes_w<W>(L.nbf, c, fs);
        T d[W], zt[W];
        widened(zv, zt);
        widened(dv, d);
#pragma unroll
        for (int t = 0; t < W; ++t) d[t] = fma(-beta, d[t], zt[t]);
        narrowed(d, dv);
        VecW<TZ, W>::store(dp, c, dv);
        if constexpr (sizeof(C) == 8) {
            double u[W];
            VecW<double, W>::load_rw(p, c, u);
#pragma unroll
            for (int t = 0; t < W; ++t)
                if (!is_solid(fs[t])) u[t] = fma(alpha, d[t], u[t]);
            VecW<double, W>::store(p, c, u);
        } else {
            float wide[W];   // alpha d where it is formed in a wider type (else at its use: one multiply-add)
            if constexpr (sizeof(T) > sizeof(C)) {
#pragma unroll
                for (int t = 0; t < W; ++t) d[t] *= alpha;
                narrowed(d, wide);
            }
            auto step = [&](int t) -> float {
                if constexpr (sizeof(T) > sizeof(C)) return wide[t];
                else return alpha * d[t];
            };
            float4* pp = reinterpret_cast<float4*>(p + c);   // p as double-float pairs, two cells per 16 bytes
#pragma unroll
            for (int h = 0; h < W / 2; ++h) {
                float4 u = pp[h];
                if (!codes || !is_solid(fs[2 * h])) {
                    const float2 x = pp_plus(make_float2(u.x, u.y), step(2 * h));
                    u.x = x.x;
                    u.y = x.y;
                }
                if (!codes || !is_solid(fs[2 * h + 1])) {
                    const float2 x = pp_plus(make_float2(u.z, u.w), step(2 * h + 1));
                    u.z = x.x;
                    u.w = x.y;
                }
                pp[h] = u;
            }
        }
    }
};
// Trilinear prolongation and correction, W consecutive x cells per thread (4 or
// 8): a lane's fine cells have the H = W/2 coarse parents I0 = i/2 .. I0 + H - 1
// (one load per coarse row).  The four coarse rows around the fine row (parent
// and neighbour along y and z, ghosts signed) are combined with their y-z
// weights first, then interpolated along x, the x neighbours I0 - 1 and I0 + H
// coming from the adjacent lanes.  Per fine cell and axis the weights are 3/4
// for the parent and 1/4 for the neighbour on the cell's side (Eq.
// prolongation); a neighbour beyond a domain face is the coarse cell's ghost,
// as in prolong_at.  Needs the x and y axes active and nx % W = 0.
template <class TI, int W>
struct ProlongVK {
    static constexpr int kThreads = TX * TY;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    static constexpr int kMinBlocks = 4;
    LevelDev Lf, Lc;
    const TI* ec;
    TI* e;
    const SolveState* st;
    int zc;    // planes per block
    int lrl;   // log2 of the lanes per row segment (as in SweepVK)
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ void run(const BlockAt& at) const;
};

// a coarse value across a ghost row or plane: negated for each zero-value face among them
template <class C>
__device__ __forceinline__ C ghost_signed(uint32_t code, bool gy, int sy, bool gz, int sz, C v) {
    bool neg = gy && ((code >> (2 * (2 + sy))) & 3u) == 2u;
    neg ^= gz && ((code >> (2 * (4 + sz))) & 3u) == 2u;
    return neg ? -v : v;
}

template <class TI, int W>
__device__ void ProlongVK<TI, W>::run(const BlockAt& at) const {
    using C = typename Acc<TI>::type;
    constexpr int H = W / 2;   // coarse cells under a thread's W fine cells
    using RC = RawW<TI, H>;
    const int nx = Lf.n[0], ny = Lf.n[1], nz = Lf.n[2];
    const int NX = Lc.n[0], NY = Lc.n[1], NZ = Lc.n[2];
    const int LR = 1 << lrl, lane = threadIdx.x & (LR - 1), sub = threadIdx.x >> lrl;
    const int i4 = at.b.x * (W * LR) + lane * W, j = ((at.b.y * TY + threadIdx.y) << (5 - lrl)) + sub;
    const int k0 = at.b.z * zc, k1 = min(nz, k0 + zc);
    const bool in = i4 < nx && j < ny;
    const bool last = i4 + W >= nx;   // the row's last coarse cell is this thread's: its x+ neighbour is a ghost
    const int ic = min(i4, nx - W), jc = min(j, ny - 1);
    const bool first = ic == 0;       // and its first: the x- neighbour is a ghost
    const int I0 = ic >> 1;
    // the y neighbour of the parent row; beyond a domain face it is the ghost row (the parent
    // row's cells, each signed by its own face code)
    const int Pj = jc >> 1, qj = Pj + ((jc & 1) ? 1 : -1);
    const bool outJ = qj < 0 || qj >= NY;
    const int Qj = outJ ? Pj : qj, sJ = qj < 0 ? 0 : 1;
    const bool zact = Lf.active[2] != 0;
    const TI* const ecp = ec;
    TI* const ep = e;
    const uint16_t* const nbf = Lf.nbf;
    const uint16_t* const cnbf = Lc.nbf;
    for (int k = k0; k < k1; ++k) {
        const int Pk = zact ? (k >> 1) : k;
        const int qk = zact ? Pk + ((k & 1) ? 1 : -1) : k;
        const bool outK = qk < 0 || qk >= NZ;
        const int Qk = outK ? Pk : qk, sK = qk < 0 ? 0 : 1;
        const C wz0 = zact ? (C)0.75 : (C)1, wz1 = zact ? (C)0.25 : (C)0;
        // the four coarse rows (parent and neighbour along y and z, ghosts signed) combined with
        // their y-z weights into one row first, then the x interpolation and the shuffles once
        C cvc[H], lc = (C)0, rc = (C)0, lg = (C)0, rg = (C)0;
#pragma unroll
        for (int h = 0; h < H; ++h) cvc[h] = (C)0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if ((q & 2) && !zact) continue;   // (a collapsed z axis: no second plane)
            const int jj = (q & 1) ? Qj : Pj, kk = (q & 2) ? Qk : Pk;
            const bool gy = (q & 1) && outJ, gz = (q & 2) && outK;
            const C w = ((q & 1) ? (C)0.25 : (C)0.75) * ((q & 2) ? wz1 : wz0);
            const int row = NX * (jj + NY * kk);
            const typename RC::T raw = RC::load(ecp, row + I0);
            C cv[H];
#pragma unroll
            for (int h = 0; h < H; ++h) cv[h] = RC::get(raw, h);
            C lft = lane == 0 ? to_c<C>(ldg(ecp + row + max(I0 - 1, 0))) : (C)0;
            C rgt = lane == LR - 1 ? to_c<C>(ldg(ecp + row + min(I0 + H, NX - 1))) : (C)0;
            uint32_t cw[H];   // the codes of the coarse cells (only where a ghost is formed)
#pragma unroll
            for (int h = 0; h < H; ++h) cw[h] = 0u;
            if (gy || gz || first || last) codes_w<H>(cnbf, row + I0, cw);
            if (gy || gz) {
#pragma unroll
                for (int h = 0; h < H; ++h) cv[h] = ghost_signed(cw[h], gy, sJ, gz, sK, cv[h]);
                if (lane == 0 && !first) lft = ghost_signed(__ldg(cnbf + row + I0 - 1), gy, sJ, gz, sK, lft);
                if (lane == LR - 1 && !last) rgt = ghost_signed(__ldg(cnbf + row + I0 + H), gy, sJ, gz, sK, rgt);
            }
#pragma unroll
            for (int h = 0; h < H; ++h) cvc[h] = fma(w, cv[h], cvc[h]);
            lc = fma(w, lft, lc);
            rc = fma(w, rgt, rc);
            if (first) lg = fma(w, (cw[0] & 3u) == 2u ? -cv[0] : cv[0], lg);                       // x- ghost of I0
            if (last) rg = fma(w, ((cw[H - 1] >> 2) & 3u) == 2u ? -cv[H - 1] : cv[H - 1], rg);   // x+ of the last
        }
        C left = __shfl_up_sync(0xffffffffu, cvc[H - 1], 1, LR);
        C right = __shfl_down_sync(0xffffffffu, cvc[0], 1, LR);
        if (lane == 0) left = lc;
        if (lane == LR - 1) right = rc;
        if (first) left = lg;
        if (last) right = rg;
        C add[W];
#pragma unroll
        for (int t = 0; t < W; ++t) {
            const int h = t >> 1;
            const C nb = (t & 1) ? (h == H - 1 ? right : cvc[h + 1]) : (h == 0 ? left : cvc[h - 1]);
            add[t] = (C)0.75 * cvc[h] + (C)0.25 * nb;
        }
        if (in) {
            const int c = ic + nx * (jc + ny * k);
            C v[W];
            uint32_t fs[W];
            VecW<TI, W>::load_rw(ep, c, v);
            GroupFlags gf = {true, false, false};
            if constexpr (sizeof(C) == 4) gf = group_flags<W>(Lf.grp, c);
            const bool codes = gf.codes;
            if (codes) codes_w<W>(nbf, c, fs);
#pragma unroll
            for (int t = 0; t < W; ++t)
                if (!codes || !is_solid(fs[t])) v[t] += add[t];
            VecW<TI, W>::store(ep, c, v);
        }
    }
}

// Residual and restriction, W x cells per thread: a thread owns the fine
// cells i4..i4+W-1 of rows 2J, 2J+1 and planes 2K, 2K+1 (2D: plane K) and
// writes the W/2 coarse cells I0 = i4/2 .. (mean of their children's r - A e,
// Eq. restriction).  Rows j +- 1 and planes k +- 1 are loaded whole, x
// neighbours by shuffles.  Needs x and y active, nx % W = 0, ny even.
template <class TI, int W, int F>   // F: kCodes, kFlags or kByLevel
struct RRVK {
    static constexpr int kThreads = TX * TY;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    static constexpr int kMinBlocks = 4;
    LevelDev Lf, Lc;
    const TI* e;
    const TI* r;
    TI* rc;
    TI* ec0;   // the coarse level's first sweep, or null
    int lrl;   // log2 of the lanes per row segment (as in SweepVK)
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ void run(const BlockAt& at) const;
};

template <class TI, int W, int F>
__device__ void RRVK<TI, W, F>::run(const BlockAt& at) const {
    using C = typename Acc<TI>::type;
    using R = RawW<TI, W>;
    constexpr int H = W / 2;
    const int nx = Lf.n[0], ny = Lf.n[1], nz = Lf.n[2];
    const int NX = Lc.n[0], NY = Lc.n[1];
    const int LR = 1 << lrl, lane = threadIdx.x & (LR - 1), sub = threadIdx.x >> lrl;
    const int i4 = at.b.x * (W * LR) + lane * W, J = ((at.b.y * TY + threadIdx.y) << (5 - lrl)) + sub, K = at.b.z;
    const bool in = i4 < nx && J < NY;
    const bool last = i4 + W >= nx;
    const int fz = Lf.active[2] ? 2 : 1;
    const int ic = min(i4, nx - W), Jc = min(J, NY - 1);
    const int ja = 2 * Jc, jb = ja + 1, jm = max(ja - 1, 0), jp = min(jb + 1, ny - 1);
    const int sy = nx, sz = nx * ny;
    const C ihx = LP<C>::ih2a(Lf, 0), ihy = LP<C>::ih2a(Lf, 1), ihz = LP<C>::ih2a(Lf, 2);
    const C dg = LP<C>::diag(Lf);
    const TI* const ep = e;
    const TI* const rp = r;
    const uint16_t* const nbf = Lf.nbf;
    const bool flags = takes_flags<F>(Lf);
    auto at_ = [&](int jj, int kk) { return ic + sy * jj + sz * kk; };
    C s[H];   // sums of the coarse cells I0 .. I0 + H - 1
#pragma unroll
    for (int h = 0; h < H; ++h) s[h] = (C)0;
    for (int dz = 0; dz < fz; ++dz) {
        const int k = fz * K + dz;
        const int km = max(k - 1, 0), kp = min(k + 1, nz - 1);
#pragma unroll
        for (int row = 0; row < 2; ++row) {
            const int jr = row ? jb : ja;
            const typename R::T ec = R::load(ep, at_(jr, k));
            const typename R::T yl = R::load(ep, at_(row ? ja : jm, k));   // row below
            const typename R::T yh = R::load(ep, at_(row ? jp : jb, k));   // row above
            const typename R::T zl = R::load(ep, at_(jr, km));
            const typename R::T zh = R::load(ep, at_(jr, kp));
            const typename R::T rr = R::load(rp, at_(jr, k));
            uint32_t fs[W];
            GroupFlags gf = {true, false, false};
            if (flags) gf = group_flags<W>(Lf.grp, at_(jr, k));
            if (gf.codes) codes_w<W>(nbf, at_(jr, k), fs);
            const C lx = lane == 0 ? to_c<C>(ldg(ep + max(ic - 1, 0) + sy * jr + sz * k)) : (C)0;
            const C rx = lane == LR - 1 ? to_c<C>(ldg(ep + min(ic + W, nx - 1) + sy * jr + sz * k)) : (C)0;
            C left = __shfl_up_sync(0xffffffffu, R::get(ec, W - 1), 1, LR);
            C right = __shfl_down_sync(0xffffffffu, R::get(ec, 0), 1, LR);
            if (lane == 0) left = lx;
            if (lane == LR - 1) right = rx;
            if (last) right = R::get(ec, W - 1);
            if constexpr (F != kCodes) {   // (at a row's ends left / right is the cell itself)
                if (gf.neg_l) left = -left;
                if (gf.neg_r) right = -right;
            }
#pragma unroll
            for (int t = 0; t < W; ++t) {
                if ((F == kCodes || gf.codes) && is_solid(fs[t])) continue;
                const C eP = R::get(ec, t);
                const C xm = t == 0 ? left : R::get(ec, t - 1), xp = t == W - 1 ? right : R::get(ec, t + 1);
                const C ya = R::get(yl, t), yb = R::get(yh, t), za = R::get(zl, t), zb = R::get(zh, t);
                if constexpr (sizeof(C) == 8) {
                    s[t >> 1] += resid64(fs[t], R::get(rr, t), eP, xm, xp, ya, yb, za, zb, ihx, ihy, ihz, dg);
                    continue;
                }
                C A;
                if ((F != kCodes && !gf.codes) || !((fs[t] >> 13) & 1u)) {
                    C sa = (xm + xp) * ihx;
                    sa = fma(ya + yb, ihy, sa);
                    sa = fma(za + zb, ihz, sa);
                    A = fma(dg, eP, -sa);
                } else {
                    A = A7_general<C>(Lf, fs[t], eP, xm, xp, ya, yb, za, zb);
                }
                s[t >> 1] += R::get(rr, t) - A;
            }
        }
    }
    if (in) {
        const C inv = (C)1 / (C)(4 * fz);
        const int o = (ic >> 1) + NX * (Jc + NY * K);
#pragma unroll
        for (int h = 0; h < H; ++h) store_restricted<TI, C>(Lc, rc, ec0, o + h, s[h] * inv);
    }
}

// coarse r = mean of the children's (r - A e): one thread per fine cell (the
// z pair of children in the thread), x / y pairs summed through shared memory.
// Needs x and y active (2 x 2 children in the plane).
template <class TI>
struct RRWalkK {
    static constexpr int kThreads = TX * TY;
    LevelDev Lf, Lc;
    const TI* e;
    const TI* r;
    TI* rc;
    TI* ec0;   // the coarse level's first sweep, or null
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }   // batched: skip a converged case
    __device__ void run(const BlockAt& at) const;
};

template <class TI>
__device__ void RRWalkK<TI>::run(const BlockAt& at) const {
    using C = typename Acc<TI>::type;
    __shared__ C part[TY][TX + 1];
    const int fz = Lf.active[2] ? 2 : 1;
    Walk w;
    const bool in = walk_setup(Lf, at, fz, w);
    C sum = (C)0;
    if (in) {
        const int nz = Lf.n[2];
        int c = w.i + w.sy * w.j + w.sz * w.k0;
        for (int kk = 0; kk < fz; ++kk) {
            const int k = w.k0 + kk;
            const uint32_t f = Lf.nbf[c];
            const C eP = to_c<C>(ldg(e + c));
            const C zm = k > 0 ? to_c<C>(ldg(e + c - w.sz)) : eP;
            const C zp = k < nz - 1 ? to_c<C>(ldg(e + c + w.sz)) : eP;
            const C xm = to_c<C>(ldg(e + c + w.im)), xp = to_c<C>(ldg(e + c + w.ip));
            const C ym = to_c<C>(ldg(e + c + w.jm)), yp = to_c<C>(ldg(e + c + w.jp));
            const C rr = to_c<C>(ldg(r + c));
            if (!is_solid(f)) sum += rr - A7<C>(Lf, f, eP, xm, xp, ym, yp, zm, zp);
            c += w.sz;
        }
    }
    part[threadIdx.y][threadIdx.x] = sum;
    __syncthreads();
    if (threadIdx.x < TX / 2 && threadIdx.y < TY / 2) {
        const int I = at.b.x * (TX / 2) + threadIdx.x, J = at.b.y * (TY / 2) + threadIdx.y;
        if (I < Lc.n[0] && J < Lc.n[1]) {
            const int x = 2 * threadIdx.x, y = 2 * threadIdx.y;
            const C s4 = (part[y][x] + part[y][x + 1]) + (part[y + 1][x] + part[y + 1][x + 1]);
            store_restricted<TI, C>(Lc, rc, ec0, I + Lc.n[0] * (J + Lc.n[1] * (int)at.b.z), s4 / (C)(4 * fz));
        }
    }
}

// ------------------------------------------------------------------ flexible CG acceleration (krylov = 1)
// One pass over level 0 with z (the V-cycles' correction for the outer
// residual r) and the kept direction d_prev: A z at each cell from the
// stencil (not stored) and the block sums of (z, A z), (A z, d_prev),
// (r, z), (r, d_prev).  The last block sums them in a fixed order and sets,
// for d = z - beta d_prev,
//   beta   = (A z, d_prev) / (d_prev, A d_prev)   [= (z, A d_prev): A is symmetric]
//   (d, A d) = (z, A z) - beta (A z, d_prev)
//   alpha  = ((r, z) - beta (r, d_prev)) / (d, A d),
// keeping (d, A d) for the next iteration.  Should rounding make (d, A d)
// non-positive (never in exact arithmetic) the direction restarts: beta = 0.
template <class TR, class TZ>
struct FcgDotK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr int kMinBlocks = 4;
    LevelDev L;
    const TZ* z;
    const TR* r;
    const TZ* dp;
    double* partials;
    SolveState* st;
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const;
};

template <class TR, class TZ>
__device__ void FcgDotK<TR, TZ>::run(const BlockAt& at) const {
    using C = typename Acc<TZ>::type;
    const bool have = st->g_valid != 0;
    double s[4] = {0.0, 0.0, 0.0, 0.0};   // (z,Az), (Az,dp), (r,z), (r,dp)
    int i, j, k;
    if (cell3(L, at, i, j, k)) {
        const int c = i + L.n[0] * (j + L.n[1] * k);
        const uint32_t f = L.nbf[c];
        const int sy = L.n[0], sz = L.n[0] * L.n[1];
        const C eP = to_c<C>(ldg(z + c));
        const C xm = to_c<C>(ldg(z + c - (i > 0 ? 1 : 0))), xp = to_c<C>(ldg(z + c + (i < L.n[0] - 1 ? 1 : 0)));
        const C ym = to_c<C>(ldg(z + c - (j > 0 ? sy : 0))), yp = to_c<C>(ldg(z + c + (j < L.n[1] - 1 ? sy : 0)));
        const C zm = to_c<C>(ldg(z + c - (k > 0 ? sz : 0))), zp = to_c<C>(ldg(z + c + (k < L.n[2] - 1 ? sz : 0)));
        const double rd = to_c<double>(ldg(r + c));
        const double dd = have ? to_c<double>(ldg(dp + c)) : 0.0;
        if (!is_solid(f)) {
            const double zd = (double)eP;
            const double qd = (double)A7<C>(L, f, eP, xm, xp, ym, yp, zm, zp);
            s[0] = zd * qd;
            s[1] = qd * dd;
            s[2] = rd * zd;
            s[3] = rd * dd;
        }
    }
    fcg_reduce<kThreads>(s, partials, st, have, at);
}

// d = z - beta d_prev; p += alpha d on fluid cells; d kept as d_prev
template <class TZ>
struct FcgUpdK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev L;
    const TZ* z;
    TZ* dp;
    double* p;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const {
        int i, j, k;
        if (!cell3(L, at, i, j, k)) return;
        const int c = i + L.n[0] * (j + L.n[1] * k);
        const double alpha = st->g_alpha, beta = st->g_beta;
        const double d = to_c<double>(ldg(z + c)) - (beta != 0.0 ? beta * to_c<double>(dp[c]) : 0.0);
        if (!is_solid(L.nbf[c])) {
            if constexpr (sizeof(TZ) == 8) p[c] += alpha * d;
            else pp_add(p, c, (float)(alpha * d));
        }
        dp[c] = from_c<TZ, double>(d);
    }
};

// ------------------------------------------------------------------ the paper's scheme (Algorithm 1)
// coarse r = mean of the children's r (the residual restricted straight down)
template <class TI>
struct RestrictK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev Lf, Lc;
    const TI* r;
    TI* rc;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const {
        using C = typename Acc<TI>::type;
        int I, J, K;
        if (!cell3(Lc, at, I, J, K)) return;
        const int fx = Lf.active[0] ? 2 : 1, fy = Lf.active[1] ? 2 : 1, fz = Lf.active[2] ? 2 : 1;
        C sum = (C)0;
        for (int dz = 0; dz < fz; ++dz)
            for (int dy = 0; dy < fy; ++dy)
                for (int dx = 0; dx < fx; ++dx)
                    sum += to_c<C>(ldg(r + (I * fx + dx) + Lf.n[0] * ((J * fy + dy) + Lf.n[1] * (K * fz + dz))));
        rc[I + Lc.n[0] * (J + Lc.n[1] * K)] = from_c<TI, C>(sum / (C)(fx * fy * fz));
    }
};

__device__ __forceinline__ int parent_of(const LevelDev& Lf, const LevelDev& Lc, int i, int j, int k) {
    const int I = Lf.active[0] ? i >> 1 : i, J = Lf.active[1] ? j >> 1 : j, K = Lf.active[2] ? k >> 1 : k;
    return I + Lc.n[0] * (J + Lc.n[1] * K);
}

// e = the parent's correction (nearest upsampling), zero in solid cells
template <class TI>
struct ProlongNearestK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev Lf, Lc;
    const TI* ec;
    TI* e;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const {
        int i, j, k;
        if (!cell3(Lf, at, i, j, k)) return;
        const int c = i + Lf.n[0] * (j + Lf.n[1] * k);
        e[c] = is_solid(Lf.nbf[c]) ? from_c<TI, float>(0.f) : ec[parent_of(Lf, Lc, i, j, k)];
    }
};

// p += the parent's level-1 correction (nearest upsampling) in fluid cells
template <class TI>
struct ProlongNearestToPK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev Lf, Lc;
    const TI* ec;
    double* p;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const {
        int i, j, k;
        if (!cell3(Lf, at, i, j, k)) return;
        const int c = i + Lf.n[0] * (j + Lf.n[1] * k);
        if (is_solid(Lf.nbf[c])) return;
        if constexpr (sizeof(TI) == 8) p[c] += to_c<double>(ldg(ec + parent_of(Lf, Lc, i, j, k)));
        else pp_add(p, c, to_c<float>(ldg(ec + parent_of(Lf, Lc, i, j, k))));
    }
};

// unweighted Jacobi sweep on the pressure, out of place: q = p + (b - A p) / D (copied back by CopyPK,
// eight bytes per cell in either storage)
template <class TB>
struct JacobiPK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev L;
    const double* p;
    const TB* b;
    double* q;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const {
        int i, j, k;
        if (!cell3(L, at, i, j, k)) return;
        const int c = i + L.n[0] * (j + L.n[1] * k);
        const uint32_t f = L.nbf[c];
        if (is_solid(f)) {
            q[c] = 0.0;
            return;
        }
        // (reduced-precision cases: p and q as double-float pairs, the sweep in FP64)
        auto P = [&](int x) { return sizeof(TB) == 8 ? __ldg(p + x) : pp_get(p, x); };
        const int sy = L.n[0], sz = L.n[0] * L.n[1];
        const double pP = P(c);
        const double xm = P(c - (i > 0 ? 1 : 0)), xp = P(c + (i < L.n[0] - 1 ? 1 : 0));
        const double ym = P(c - (j > 0 ? sy : 0)), yp = P(c + (j < L.n[1] - 1 ? sy : 0));
        const double zm = P(c - (k > 0 ? sz : 0)), zp = P(c + (k < L.n[2] - 1 ? sz : 0));
        const double v = pP + (to_c<double>(ldg(b + c)) - A7<double>(L, f, pP, xm, xp, ym, yp, zm, zp)) * L.inv_D;
        if constexpr (sizeof(TB) == 8) q[c] = v;
        else reinterpret_cast<float2*>(q)[c] = pp_from_double(v);
    }
};

struct CopyPK {
    static constexpr int kThreads = BX * BY * BZ;
    static constexpr bool kNoShared = true;   // run() uses no shared memory
    LevelDev L;
    const double* q;
    double* p;
    const SolveState* st;
    __device__ bool live() const { return st->active != 0; }
    __device__ void run(const BlockAt& at) const {
        int i, j, k;
        if (!cell3(L, at, i, j, k)) return;
        const int c = i + L.n[0] * (j + L.n[1] * k);
        p[c] = q[c];
    }
};

__global__ void k_p_to_double(const double* __restrict__ pp, double* __restrict__ dst, int64_t N) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < N) dst[c] = pp_get(pp, c);
}

__global__ void k_p_from_double(const double* __restrict__ src, double* __restrict__ pp, int64_t N) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < N) reinterpret_cast<float2*>(pp)[c] = pp_from_double(src[c]);
}

// p to and from FP32 host values: the pair rounded once to FP32 (hi + lo evaluated in FP64,
// exact), and an FP32 value as the pair (value, 0)
__global__ void k_p_to_float(const double* __restrict__ pp, float* __restrict__ dst, int64_t N) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < N) dst[c] = __double2float_rn(pp_get(pp, c));
}

__global__ void k_p_from_float(const float* __restrict__ src, double* __restrict__ pp, int64_t N) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < N) reinterpret_cast<float2*>(pp)[c] = make_float2(src[c], 0.0f);
}

template <class A, class B>
__global__ void k_convert(const A* __restrict__ src, B* __restrict__ dst, int64_t N) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < N) dst[c] = from_c<B, double>(to_c<double>(src[c]));
}

dim3 grid3(const LevelDev& L) {
    return dim3((unsigned)((L.n[0] + BX - 1) / BX), (unsigned)((L.n[1] + BY - 1) / BY),
                (unsigned)((L.n[2] + BZ - 1) / BZ));
}
const dim3 kBlock3(BX, BY, BZ);

}  // namespace

int resid0_blocks(int nx, int ny, int nz) {
    return ((nx + BX - 1) / BX) * ((ny + BY - 1) / BY) * ((nz + BZ - 1) / BZ);
}

// vector kernels with W cells per thread: log2 of the lanes per row segment, the widest
// segment of W * 32, W * 16, W * 8 or W * 4 cells that divides nx (a warp then covers 1, 2, 4
// or 8 rows)
static int vw_lrl(int nx, int W) {
    for (int l = 5; l >= 2; --l)
        if (nx % (W << l) == 0) return l;
    return 5;
}
static int v4_lrl(int nx) { return vw_lrl(nx, 4); }

int level0_blocks_max(int nx, int ny, int nz) {
    // a vector pass (four or eight cells per thread) with this nx's row segments, one plane a block
    int most = resid0_blocks(nx, ny, nz);
    for (int W : {2, 4, 8}) {
        const int lrl = vw_lrl(nx, W), wx = W << lrl, wy = TY << (5 - lrl);
        const int n = ((nx + wx - 1) / wx) * ((ny + wy - 1) / wy) * nz;
        most = n > most ? n : most;
    }
    return most;
}

#define DISPATCH_I(inner, ...)                                            \
    do {                                                                  \
        if ((inner) == FVM_FP64) { using TI = double; __VA_ARGS__; }      \
        else if ((inner) == FVM_FP32) { using TI = float; __VA_ARGS__; } \
        else { using TI = __nv_bfloat16; __VA_ARGS__; }                   \
    } while (0)

cudaError_t launch_solve_begin(SolveState* st, cudaStream_t s) {
    return launch_k(SolveBeginK{st}, dim3(1), dim3(1), 0, s);
}

static int sweep_planes(int tiles, int nz, int fixed, int per_sm, int W, bool sums);

// vector kernels: the block's x-y extent for W cells per thread and the row segments of lrl;
// per_sm: the blocks per SM the plane rule aims for; sums: the columns order a sum
static dim3 vw_grid(const LevelDev& L, int W, int lrl, int& zc, int per_sm = 8, bool sums = false) {
    const int wx = W << lrl, wy = TY << (5 - lrl);
    const int tiles = ((L.n[0] + wx - 1) / wx) * ((L.n[1] + wy - 1) / wy);
    zc = sweep_planes(tiles, L.n[2], L.zc_fixed, per_sm, W, sums);
    return dim3((unsigned)((L.n[0] + wx - 1) / wx), (unsigned)((L.n[1] + wy - 1) / wy), (unsigned)((L.n[2] + zc - 1) / zc));
}

cudaError_t launch_resid0(int inner, int bprec, const LevelDev& L, const double* p, const void* b, void* r, void* e,
                          double* partials, SolveState* st, cudaGraphConditionalHandle cond, int use_cond,
                          cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    DISPATCH_I(inner, {
        if constexpr (sizeof(TI) < 8) {
            // four cells per thread in float-float on large levels and in batches
            if (bprec == FVM_FP32 && L.n[0] % 4 == 0 && (L.N >= (1 << 20) || g_rec)) {
                const int lrl = v4_lrl(L.n[0]);
                int zc = 0;
                const dim3 grid = vw_grid(L, 4, lrl, zc, 8, true);
                // (at most level0_blocks_max(n) blocks: partials has room)
                return by_form(L, [&](auto f) {
                    return launch_r0(Resid0V4K<TI, decltype(f)::value>{L, p, (const float*)b, (TI*)r, (TI*)e, partials, st, zc, lrl},
                                     grid, dim3(TX, TY), cond, use_cond, s);
                });
            }
        }
        // two cells per thread in FP64 on FP64 levels, and on the smaller ones of a reduced-precision
        // case alone (Resid0DK)
        using TB = std::conditional_t<sizeof(TI) == 8, double, float>;
        if (bprec == (sizeof(TI) == 8 ? FVM_FP64 : FVM_FP32) && L.n[0] % (sizeof(TI) == 8 ? 2 : 4) == 0) {
            const int lrl = vw_lrl(L.n[0], 2);
            int zc = 0;
            const dim3 grid = vw_grid(L, 2, lrl, zc, 8, true);
            return launch_r0(Resid0DK<TB, TI>{L, p, (const TB*)b, (TI*)r, (TI*)e, partials, st, zc, lrl}, grid,
                             dim3(TX, TY), cond, use_cond, s);
        }
        if (bprec == FVM_FP64)
            err = launch_r0(Resid0K<double, TI>{L, p, (const double*)b, (TI*)r, (TI*)e, partials, st}, grid3(L),
                            kBlock3, cond, use_cond, s);
        else
            err = launch_r0(Resid0K<float, TI>{L, p, (const float*)b, (TI*)r, (TI*)e, partials, st}, grid3(L),
                            kBlock3, cond, use_cond, s);
    });
    return err;
}

cudaError_t launch_sweep_first(int inner, const LevelDev& L, const void* r, void* e, const SolveState* st,
                               cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    DISPATCH_I(inner, err = launch_k(SweepFirstK<TI>{L, (const TI*)r, (TI*)e, st}, grid3(L), kBlock3, 0, s));
    return err;
}

static dim3 walk_grid(const LevelDev& L, int kz) {
    return dim3((unsigned)((L.n[0] + TX - 1) / TX), (unsigned)((L.n[1] + TY - 1) / TY),
                (unsigned)((L.n[2] + kz - 1) / kz));
}

// planes per block: the most that still give about per_sm blocks per SM (one plane per
// block on grids too small for that).  The sweep aims for 16: it has no block reduction, and
// shorter columns in more blocks balance better (the room's level-0 sweep: 42.3 us at four
// planes a block, 37.3 at two, 40.0 at one); the kernels that end in a block reduction (the
// residual, the inner products) aim for 8 at 16 planes and more, for 1000 blocks (about two
// waves) at 8, 4 and 2 planes, and take two planes rather than one from two blocks per SM on: a
// block that reduces one plane's sums costs more than a second plane (ten steps of the
// 256 x 64 x 64 FP32 channel 8.77 -> 8.19 ms from one plane to two; four of the 512 x 128 x 128
// one 12.94 -> 12.84 ms from four planes to eight; 24 cycles of a 256 x 128 x 128 BF16 room 5.70
// -> 5.60 ms from two planes to four; the 512 x 256 x 128 room at 16 planes instead of 8 54.3 ->
// 55.1 ms; at two, both kernels a third slower).
static int sweep_planes(int tiles, int nz, int fixed, int per_sm, int W, bool sums) {
    if (fixed > 0) return fixed < nz ? fixed : nz;
    auto blocks = [&](int zc) { return tiles * ((nz + zc - 1) / zc); };
    const bool reduces = per_sm <= 8;
    if (g_rec) {
        // in a batch the cases' blocks add up (taken as all of this case's size): the longest columns
        // of at most eight planes that leave the launch this many blocks, fewer for the kernels that
        // end in a block reduction and more for the eight-cell sweep (two planes of a small level's
        // block take longer than the level: with eight-plane columns throughout, 8 FP32 channels
        // took 14.8 ms for four steps against 13.6 ms, 8 served BF16 cases 43.9 against 34.0 ms for
        // two; 64 channels 19.4 ms a step either way).  Columns that order a sum are those of a batch of
        // eight in any batch (as of four, the residual of 8 channels took 77 us for 63): a case's
        // results do not depend on how many others there are
        const int want = reduces ? 300 : (W == 8 ? 1500 : 608);
        for (int zc : {8, 4, 2})
            if ((int64_t)blocks(zc) * (sums ? 8 : g_rec->cases) >= want) return nz < zc ? nz : zc;
        return 1;
    }
    for (int zc : {32, 16, 8, 4, 2})
        if (blocks(zc) >= (reduces && zc <= 8 ? 1000 : per_sm * 152)) return zc;
    return reduces && blocks(2) >= 2 * 152 ? 2 : 1;
}

// eight cells per thread on BF16 levels: in batches, and on single-case levels of 2^22 cells or
// more; a smaller level (the room's level 1, 2 M cells) takes four, for twice the threads (at
// eight its residual-restriction launch had 256 blocks for 152 SMs)
static bool wide8(const LevelDev& L) { return L.n[0] % 8 == 0 && (g_rec || L.N >= (1 << 22)); }

template <class TI, int MODE>
static cudaError_t sweep_walk(const LevelDev& L, const TI* ein, const TI* r, TI* eout, double* p,
                              const SolveState* st, cudaStream_t s, float* z32 = nullptr) {
    if constexpr (sizeof(TI) < 8) {
        // four cells per thread on large levels and in batches (their blocks add up over the cases)
        if (L.n[0] % 4 == 0 && (L.N >= (1 << 20) || g_rec)) {
            constexpr int W = vec_w<TI>();
            int zc = 0;
            if (W == 8 && wide8(L)) {
                const int lrl = vw_lrl(L.n[0], 8);
                const dim3 grid = vw_grid(L, 8, lrl, zc, 16);
                return launch_k(SweepVK<TI, MODE, vec_w<TI>()>{L, ein, r, eout, p, st, zc, z32, lrl}, grid,
                                dim3(TX, TY), 0, s);
            }
            const int lrl = vw_lrl(L.n[0], 4);
            const dim3 grid = vw_grid(L, 4, lrl, zc, 16);
            return launch_k(SweepVK<TI, MODE, 4>{L, ein, r, eout, p, st, zc, z32, lrl}, grid, dim3(TX, TY), 0, s);
        }
    }
    if constexpr (sizeof(TI) == 8 && MODE != 2) {
        if (L.n[0] % 2 == 0) {
            int zc = 0;
            const int lrl = vw_lrl(L.n[0], 2);
            const dim3 grid = vw_grid(L, 2, lrl, zc, 16);
            return launch_k(SweepVK<TI, MODE, 2>{L, ein, r, eout, p, st, zc, z32, lrl}, grid, dim3(TX, TY), 0, s);
        }
    }
    // four cells per thread on large grids and in batches (one launch for all cases of a level)
    if (L.N >= (1 << 20) || g_rec)
        return launch_k(SweepK<TI, MODE, 4>{L, ein, r, eout, p, st, z32}, walk_grid(L, 4), dim3(TX, TY), 0, s);
    return launch_k(SweepK<TI, MODE, 1>{L, ein, r, eout, p, st, z32}, walk_grid(L, 1), dim3(TX, TY), 0, s);
}

cudaError_t launch_sweep(int inner, const LevelDev& L, const void* e_in, const void* r, void* e_out,
                         const SolveState* st, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    DISPATCH_I(inner, err = sweep_walk<TI, 0>(L, (const TI*)e_in, (const TI*)r, (TI*)e_out, nullptr, st, s));
    return err;
}

cudaError_t launch_sweep_to_p(int inner, const LevelDev& L, const void* e_in, const void* r, double* p,
                              const SolveState* st, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    DISPATCH_I(inner, err = sweep_walk<TI, 1>(L, (const TI*)e_in, (const TI*)r, nullptr, p, st, s));
    return err;
}

cudaError_t launch_sweep_to_f32(int inner, const LevelDev& L, const void* e_in, const void* r, float* z,
                                const SolveState* st, cudaStream_t s) {
    if (inner != FVM_BF16_MIXED) return cudaErrorInvalidValue;
    using TI = __nv_bfloat16;
    return sweep_walk<TI, 2>(L, (const TI*)e_in, (const TI*)r, nullptr, nullptr, st, s, z);
}

template <class TI>
static bool v4_transfer_ok(const LevelDev& Lf) {
    return sizeof(TI) < 8 && Lf.active[0] && Lf.active[1] && Lf.n[0] % 4 == 0 && Lf.n[1] % 2 == 0 &&
           (Lf.N >= (1 << 20) || g_rec);
}

CodeBytes code_bytes(int inner, const LevelDev& L) {
    const double N = (double)L.N, codes = 2.0 * N, flags = N / 8.0, either = L.solids ? codes : flags;
    const bool quads = inner != FVM_FP64 && L.n[0] % 4 == 0, vector = quads && (L.N >= (1 << 20) || g_rec);
    const bool transfer = inner != FVM_FP64 && v4_transfer_ok<float>(L);
    return {vector ? flags : codes, vector ? either : codes, transfer ? either : codes, transfer ? flags : codes,
            quads ? either + flags : 2.0 * codes};
}

cudaError_t launch_resid_restrict(int inner, const LevelDev& Lf, const LevelDev& Lc, const void* e, const void* r,
                                  void* rc, void* ec0, const SolveState* st, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    if (inner != FVM_FP64 && v4_transfer_ok<float>(Lf)) {
        const int W = inner == FVM_BF16_MIXED && wide8(Lf) ? 8 : 4;
        const int lrl = vw_lrl(Lf.n[0], W), wx = W << lrl, wy = TY << (5 - lrl);
        const dim3 grid((unsigned)((Lf.n[0] + wx - 1) / wx), (unsigned)((Lc.n[1] + wy - 1) / wy), (unsigned)Lc.n[2]);
        auto go = [&](auto ti, auto w, auto f) {
            using TI = decltype(ti);
            return launch_k(RRVK<TI, decltype(w)::value, decltype(f)::value>{Lf, Lc, (const TI*)e, (const TI*)r, (TI*)rc,
                                                                             (TI*)ec0, lrl, st},
                            grid, dim3(TX, TY), 0, s);
        };
        using W4 = std::integral_constant<int, 4>;
        using W8 = std::integral_constant<int, 8>;
        if (inner == FVM_FP32) return by_form(Lf, [&](auto f) { return go(0.0f, W4(), f); });
        const __nv_bfloat16 b16{};
        if (W == 8) return by_form(Lf, [&](auto f) { return go(b16, W8(), f); });
        return by_form(Lf, [&](auto f) { return go(b16, W4(), f); });
    }
    if (inner == FVM_FP64 && Lf.active[0] && Lf.active[1]) {   // (active axes of a level that is coarsened are even)
        const int lrl = vw_lrl(Lf.n[0], 2), wx = 2 << lrl, wy = TY << (5 - lrl);
        const dim3 grid((unsigned)((Lf.n[0] + wx - 1) / wx), (unsigned)((Lc.n[1] + wy - 1) / wy), (unsigned)Lc.n[2]);
        return launch_k(RRVK<double, 2, kCodes>{Lf, Lc, (const double*)e, (const double*)r, (double*)rc, (double*)ec0, lrl, st},
                        grid, dim3(TX, TY), 0, s);
    }
    if (Lf.active[0] && Lf.active[1]) {
        const int fz = Lf.active[2] ? 2 : 1;
        auto walk = [&](auto ti) {
            using TI = decltype(ti);
            return launch_k(RRWalkK<TI>{Lf, Lc, (const TI*)e, (const TI*)r, (TI*)rc, (TI*)ec0, st}, walk_grid(Lf, fz),
                            dim3(TX, TY), 0, s);
        };
        err = inner == FVM_FP32 ? walk(0.0f) : walk(__nv_bfloat16());
    } else {
        DISPATCH_I(inner, err = launch_k(ResidRestrictK<TI>{Lf, Lc, (const TI*)e, (const TI*)r, (TI*)rc, (TI*)ec0,
                                                            st},
                                         grid3(Lc), kBlock3, 0, s));
    }
    return err;
}

cudaError_t launch_prolong_add(int inner, const LevelDev& Lf, const LevelDev& Lc, const void* ec, void* e,
                               const SolveState* st, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    if (inner != FVM_FP64 && v4_transfer_ok<float>(Lf)) {
        int zc = 0;
        if (inner == FVM_FP32) {
            const int lrl = vw_lrl(Lf.n[0], 4);
            const dim3 grid = vw_grid(Lf, 4, lrl, zc);
            return launch_k(ProlongVK<float, 4>{Lf, Lc, (const float*)ec, (float*)e, st, zc, lrl}, grid, dim3(TX, TY),
                            0, s);
        }
        if (wide8(Lf)) {
            const int lrl = vw_lrl(Lf.n[0], 8);
            const dim3 grid = vw_grid(Lf, 8, lrl, zc);
            return launch_k(ProlongVK<__nv_bfloat16, 8>{Lf, Lc, (const __nv_bfloat16*)ec, (__nv_bfloat16*)e, st, zc,
                                                        lrl},
                            grid, dim3(TX, TY), 0, s);
        }
        const int lrl = vw_lrl(Lf.n[0], 4);
        const dim3 grid = vw_grid(Lf, 4, lrl, zc);
        return launch_k(ProlongVK<__nv_bfloat16, 4>{Lf, Lc, (const __nv_bfloat16*)ec, (__nv_bfloat16*)e, st, zc, lrl},
                        grid, dim3(TX, TY), 0, s);
    }
    if (inner == FVM_FP64 && Lf.active[0] && Lf.active[1]) {
        int zc = 0;
        const int lrl = vw_lrl(Lf.n[0], 2);
        const dim3 grid = vw_grid(Lf, 2, lrl, zc);
        return launch_k(ProlongVK<double, 2>{Lf, Lc, (const double*)ec, (double*)e, st, zc, lrl}, grid, dim3(TX, TY), 0, s);
    }
    DISPATCH_I(inner, err = launch_k(ProlongK<TI>{Lf, Lc, (const TI*)ec, (TI*)e, st}, grid3(Lf), kBlock3, 0, s));
    return err;
}

// z and the kept direction dp in TZ (the inner type, or FP32 on BF16 levels), r in TR: W cells per
// thread, products, sums and the step in T
template <class TR, class TZ, int W, class T>
static cudaError_t fcg_vector(const LevelDev& L, const TZ* z, const TR* r, TZ* dp, double* p, double* partials,
                              SolveState* st, cudaStream_t s) {
    // (at most level0_blocks_max(n) blocks: partials has room)
    int zc = 0;
    const int lrl = vw_lrl(L.n[0], W);
    const dim3 grid = vw_grid(L, W, lrl, zc, 8, true);
    auto dot = [&](auto f) {
        return launch_k(FcgDotVK<TR, TZ, W, decltype(f)::value, T>{L, z, r, dp, partials, st, zc, lrl}, grid, dim3(TX, TY), 0, s);
    };
    cudaError_t err;
    if constexpr (sizeof(TZ) == 8) err = dot(std::integral_constant<int, kCodes>());
    else err = by_form(L, dot);
    if (err != cudaSuccess) return err;
    using U = FcgUpdVK<TZ, W, T>;
    return launch_k(U{L, z, dp, p, st}, dim3((unsigned)((L.N / W + U::kThreads - 1) / U::kThreads)), dim3(U::kThreads), 0, s);
}

template <class TR, class TZ>
static cudaError_t fcg_launch(const LevelDev& L, const TZ* z, const TR* r, TZ* dp, double* p, double* partials,
                              SolveState* st, cudaStream_t s) {
    if constexpr (sizeof(TR) < 8) {
        if (L.n[0] % 4 == 0) {
            // products, sums, alpha and beta in FP32 on large levels and in batches; in FP64 on the smaller
            // ones of a case alone (430,080 cells, us for the pair of launches: one cell per thread 58, this
            // 35, the FP32 form 22)
            if (L.N < (1 << 20) && !g_rec) return fcg_vector<TR, TZ, 4, double>(L, z, r, dp, p, partials, st, s);
            constexpr int W = std::is_same<TR, TZ>::value ? vec_w<TR>() : 4;
            if (L.n[0] % W == 0) return fcg_vector<TR, TZ, W, float>(L, z, r, dp, p, partials, st, s);
            return fcg_vector<TR, TZ, 4, float>(L, z, r, dp, p, partials, st, s);
        }
    }
    if constexpr (sizeof(TR) == 8) {
        if (L.n[0] % 2 == 0) return fcg_vector<TR, TZ, 2, double>(L, z, r, dp, p, partials, st, s);
    }
    cudaError_t err = launch_k(FcgDotK<TR, TZ>{L, z, r, dp, partials, st}, grid3(L), kBlock3, 0, s);
    if (err != cudaSuccess) return err;
    return launch_k(FcgUpdK<TZ>{L, z, dp, p, st}, grid3(L), kBlock3, 0, s);
}

cudaError_t launch_fcg(int inner, const LevelDev& L, const void* z, const void* r, void* dp, double* p,
                       double* partials, SolveState* st, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    if (inner == FVM_BF16_MIXED)   // z and the kept direction in FP32 (rounding them to BF16 costs V-cycles)
        return fcg_launch<__nv_bfloat16, float>(L, (const float*)z, (const __nv_bfloat16*)r, (float*)dp, p, partials,
                                                st, s);
    DISPATCH_I(inner, err = fcg_launch<TI, TI>(L, (const TI*)z, (const TI*)r, (TI*)dp, p, partials, st, s));
    return err;
}

cudaError_t launch_restrict(int inner, const LevelDev& Lf, const LevelDev& Lc, const void* r, void* rc,
                            const SolveState* st, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    DISPATCH_I(inner, err = launch_k(RestrictK<TI>{Lf, Lc, (const TI*)r, (TI*)rc, st}, grid3(Lc), kBlock3, 0, s));
    return err;
}

cudaError_t launch_prolong_nearest(int inner, const LevelDev& Lf, const LevelDev& Lc, const void* ec, void* e,
                                   const SolveState* st, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    DISPATCH_I(inner, err = launch_k(ProlongNearestK<TI>{Lf, Lc, (const TI*)ec, (TI*)e, st}, grid3(Lf), kBlock3, 0, s));
    return err;
}

cudaError_t launch_prolong_nearest_to_p(int inner, const LevelDev& Lf, const LevelDev& Lc, const void* ec, double* p,
                                        const SolveState* st, cudaStream_t s) {
    cudaError_t err = cudaSuccess;
    DISPATCH_I(inner,
               err = launch_k(ProlongNearestToPK<TI>{Lf, Lc, (const TI*)ec, p, st}, grid3(Lf), kBlock3, 0, s));
    return err;
}

cudaError_t launch_jacobi_p(int bprec, const LevelDev& L, double* p, const void* b, double* q, const SolveState* st,
                            cudaStream_t s) {
    cudaError_t err;
    if (bprec == FVM_FP64) err = launch_k(JacobiPK<double>{L, p, (const double*)b, q, st}, grid3(L), kBlock3, 0, s);
    else err = launch_k(JacobiPK<float>{L, p, (const float*)b, q, st}, grid3(L), kBlock3, 0, s);
    if (err != cudaSuccess) return err;
    return launch_k(CopyPK{L, q, p, st}, grid3(L), kBlock3, 0, s);
}

cudaError_t launch_convert(int sp, int dp, const void* src, void* dst, int64_t N, cudaStream_t s) {
    const unsigned nb = (unsigned)((N + 255) / 256);
    if (sp == FVM_FP64 && dp == FVM_FP32) k_convert<double, float><<<nb, 256, 0, s>>>((const double*)src, (float*)dst, N);
    else if (sp == FVM_FP32 && dp == FVM_FP64) k_convert<float, double><<<nb, 256, 0, s>>>((const float*)src, (double*)dst, N);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_p_to_double(const double* pp, double* dst, int64_t N, cudaStream_t s) {
    k_p_to_double<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(pp, dst, N);
    return cudaGetLastError();
}

cudaError_t launch_p_to_float(const double* pp, float* dst, int64_t N, cudaStream_t s) {
    k_p_to_float<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(pp, dst, N);
    return cudaGetLastError();
}

cudaError_t launch_p_from_float(const float* src, double* pp, int64_t N, cudaStream_t s) {
    k_p_from_float<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(src, pp, N);
    return cudaGetLastError();
}

cudaError_t launch_p_from_double(const double* src, double* pp, int64_t N, cudaStream_t s) {
    k_p_from_double<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(src, pp, N);
    return cudaGetLastError();
}
