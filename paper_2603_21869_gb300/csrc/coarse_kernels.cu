// The multigrid levels below the grid-wide ones (on a small grid with plain V-cycles, all of them), in
// one thread-block cluster per V-cycle.
//
// A level of a few thousand to some ten thousand cells keeps no GPU busy: run as one launch per
// sweep or transfer, each launch is a chain of latencies (parameters, face codes, neighbour loads,
// store, the next launch), 4-5 us whatever the level's size, and the smallest levels on one SM
// alone wait for that SM's issue slots and, at the coarsest level, for one SM to read the dense
// inverse (4 MB at 1024 unknowns).  Here up to 16 SMs hold the levels' corrections in their shared
// memory for the whole down and up sweep: a level's planes along its outermost active axis are
// dealt to the blocks of the cluster in equal contiguous slabs, a sweep reads the two planes beyond
// a slab from the neighbouring blocks' shared memory (distributed shared memory), and phases are
// separated by the hardware cluster barrier (0.24 us at 16 blocks of 512 threads, measured).
// Levels too small to deal out run on block 0 between CTA barriers, and the dense coarsest solve
// is shared out by rows.  What bounds it: the latency of each phase (shared-memory loads, the
// neighbouring blocks' planes, the barrier).  A sweep takes 0.5 us on block 0, 0.9-1.1 us dealt out
// at up to 1024 cells a block, 1.9 us at 4096.  Per V-cycle, against one SM for the coarse levels and
// launches for the others: the levels of 65,536 cells and below of a 256 x 128 x 128 room 33 us
// against 112 + 37 us, of 53,760 and below of a 112 x 80 x 48 room 27 us against 69 + 38 us.
#include <cooperative_groups.h>

#include <cstring>

#include "fvm_internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kCtaThreads = 512;

template <class T> struct Acc { using type = T; };
template <> struct Acc<__nv_bfloat16> { using type = float; };

// One level as the cluster's blocks see it.  Axis `slow` is the outermost active one: its ns
// planes of P consecutive cells belong m to a block (a level that block 0 keeps to itself: m = ns).
template <class C>
struct ClusterLevel {
    int32_t n[3], act[3];
    int32_t slow, P, ns, m;
    int32_t e0, e1, r;       // this level's arrays in the dynamic shared memory (elements of C);
                             // r < 0: r and the codes stay in global memory (the finest level of
                             // the cluster, where they do not fit)
    int32_t f;               // its codes in shared memory (16-bit units)
    uint32_t dir;            // bit d: face d has a zero-value cell on this level
    int32_t pad;
    C ih[3], diag, iD, wJ;
    const uint16_t* nbf;
};

template <class TI>
struct CoarseK {
    using C = typename Acc<TI>::type;
    int32_t S;               // blocks of the cluster
    int32_t nl, lm;          // levels; the first lm are dealt out, the rest are block 0's
    int32_t pre, post, cheb;
    int32_t dense_all;       // the coarsest solve's rows are shared out over all blocks
    int32_t x;               // offset of the coarsest right-hand side
    ClusterLevel<C> lv[FVM_MAX_LEVELS];
    C w[2][kMaxChebSweeps];  // smoother 1: the weight of sweep i before (0) and after (1) the coarse correction
    const TI* r_in;
    TI* e_out;
    double* p;               // the finest level is level 0: its correction is added to p (else null)
    const double* Ainv;
    const SolveState* st;
};

__device__ __forceinline__ bool is_solid(uint32_t f) { return (f >> 12) & 1u; }

// every thread of the cluster; release / acquire at cluster scope
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// c / n for 0 <= c < 2^22 with inv_n = 1/n in FP32: (c + 1/2)/n is at least 1/(2n) from an
// integer, more than the FP32 rounding of the product
__device__ __forceinline__ int small_div(int c, float inv_n) { return (int)(((float)c + 0.5f) * inv_n); }

// Four consecutive values (16-byte aligned)
template <class C> struct Quad { C v[4]; };
__device__ __forceinline__ Quad<float> load4(const float* p) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    return {{a.x, a.y, a.z, a.w}};
}
__device__ __forceinline__ Quad<double> load4(const double* p) {
    const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
    return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ Quad<float> load4(const __nv_bfloat16* p) {
    const uint2 a = *reinterpret_cast<const uint2*>(p);
    return {{__uint_as_float(a.x << 16), __uint_as_float(a.x & 0xffff0000u), __uint_as_float(a.y << 16),
             __uint_as_float(a.y & 0xffff0000u)}};
}
__device__ __forceinline__ void load2(const float* p, float& a, float& b) {   // (8-byte aligned)
    const float2 v = *reinterpret_cast<const float2*>(p);
    a = v.x;
    b = v.y;
}
__device__ __forceinline__ void load2(const double* p, double& a, double& b) {
    a = p[0];
    b = p[1];
}
__device__ __forceinline__ void store4(float* p, const Quad<float>& q) {
    *reinterpret_cast<float4*>(p) = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]);
}
__device__ __forceinline__ void store4(double* p, const Quad<double>& q) {
    reinterpret_cast<double2*>(p)[0] = make_double2(q.v[0], q.v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(q.v[2], q.v[3]);
}
__device__ __forceinline__ void store4(__nv_bfloat16* p, const Quad<float>& q) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(q.v[0], q.v[1]), b = __floats2bfloat162_rn(q.v[2], q.v[3]);
    uint2 u;
    memcpy(&u.x, &a, 4);
    memcpy(&u.y, &b, 4);
    *reinterpret_cast<uint2*>(p) = u;
}

// One level as this block works on it, in shared memory (one thread per level forms it at the
// start: formed by every thread at every phase it cost about half a microsecond a phase).
// Offsets are into the dynamic shared memory, in elements of C (f: in codes).
template <class C>
struct Slab {
    int32_t own, np, k0, P;  // this block's cells and planes, its first plane, cells per plane
    int32_t nx, slow;
    int32_t e0, flip;        // the two e arrays: e0 and e0 + flip
    int32_t r, f;            // < 0: r and the codes in global memory
    int32_t all;             // dealt out: phases end in a cluster barrier
    int32_t quads;           // three active axes, rows of whole quads: the four-cell forms
    int32_t x, y;            // x / y is an active axis inside a plane
    int32_t joined;          // both children planes of every coarse plane here belong to this block
    int32_t base;            // the slab's first cell in the level's arrays
    C ih[3], diag, iD, wJ;
    const C* prev;           // the plane before the slab's first and the one after its last, of the
    const C* next;           // first e array, in the neighbouring blocks (valid memory at the ends too)
    const uint16_t* nbf;     // the slab's codes in global memory
};

template <class TI>
struct Body {
    using C = typename Acc<TI>::type;
    const CoarseK<TI>& k;
    C* const sm;
    Slab<C>* const tab;      // (shared memory) the levels
    const int rank;
    const int tid, T;

    __device__ __forceinline__ Body(const CoarseK<TI>& k_, unsigned char* raw, Slab<C>* tab_, int rank_)
        : k(k_), sm(reinterpret_cast<C*>(raw)), tab(tab_), rank(rank_), tid(threadIdx.x), T(blockDim.x) {}

    __device__ __forceinline__ bool dealt(int l) const { return l < k.lm; }
    __device__ __forceinline__ const uint16_t* codes() const { return reinterpret_cast<const uint16_t*>(sm); }
    // the same array in block q's shared memory
    __device__ __forceinline__ C* at(C* p, int q) const {
        return q == rank ? p : cg::this_cluster().map_shared_rank(p, q);
    }
    __device__ __forceinline__ void barrier(bool all) const {
        if (all) cluster_barrier();
        else __syncthreads();
    }
    __device__ __forceinline__ C weight(const Slab<C>& s, int side, int i) const { return k.cheb ? k.w[side][i] : s.wJ; }

    __device__ __forceinline__ void form_slab(int l) const {
        const ClusterLevel<C>& L = k.lv[l];
        Slab<C>& s = tab[l];
        const bool d = dealt(l);
        s.np = d ? max(0, min(L.ns - rank * L.m, L.m)) : (rank == 0 ? L.ns : 0);
        s.k0 = d ? rank * L.m : 0;
        s.P = L.P;
        s.own = s.np * L.P;
        s.base = s.k0 * L.P;
        s.nx = L.slow > 0 ? L.n[0] : 1;
        s.slow = L.slow;
        s.e0 = L.e0;
        s.flip = L.e1 - L.e0;
        s.r = L.r;
        s.f = L.f;
        s.all = d;
        s.quads = L.act[0] && L.act[1] && L.act[2] && L.n[0] % 4 == 0;
        s.x = L.act[0] && L.slow > 0;
        s.y = L.act[1] && L.slow > 1;
        s.joined = l + 2 < k.nl && (d ? dealt(l + 1) && L.m == 2 * k.lv[l + 1].m : true);
        for (int a = 0; a < 3; ++a) s.ih[a] = L.ih[a];
        s.diag = L.diag;
        s.iD = L.iD;
        s.wJ = L.wJ;
        s.nbf = L.nbf + s.base;
        C* const b = sm + L.e0;
        s.prev = s.next = b;
        if (d && s.np > 0) {   // (a block without planes reads nothing)
            if (rank > 0) s.prev = at(b, rank - 1) + (L.m - 1) * L.P;
            if ((rank + 1) * L.m < L.ns) s.next = at(b, rank + 1);
        }
    }

    __device__ __forceinline__ uint32_t code(const Slab<C>& s, int c) const {
        return s.f >= 0 ? (uint32_t)codes()[s.f + c] : (uint32_t)__ldg(s.nbf + c);
    }
    __device__ __forceinline__ C rhs(const Slab<C>& s, int c) const {
        return s.r >= 0 ? sm[s.r + c] : to_c<C>(ldg(k.r_in + s.base + c));
    }
    __device__ __forceinline__ Quad<C> rhs4(const Slab<C>& s, int c) const {
        return s.r >= 0 ? load4(sm + s.r + c) : load4(k.r_in + s.base + c);
    }
    __device__ __forceinline__ uint2 codes4(const Slab<C>& s, int c) const {
        return s.f >= 0 ? *reinterpret_cast<const uint2*>(codes() + s.f + c)
                        : __ldg(reinterpret_cast<const uint2*>(s.nbf + c));
    }
    static __device__ __forceinline__ uint32_t code_of(uint2 w, int q) {
        const uint32_t v = q < 2 ? w.x : w.y;
        return (q & 1) ? v >> 16 : v & 0xffffu;
    }

    // A e of a fluid cell from its neighbours as loaded: diag e_P - sum_a ih_a (lo + hi).  A
    // neighbour across a zero-gradient face is the cell itself; a zero-value face's ghost is
    // -e_P: in FP32 the rare 2 ih_a e_P added to that, in FP64 a sign (an integer operation; a
    // second FP64 pass over a warp costs as much as the stencil).
    static constexpr bool kSigned = sizeof(C) == 8;
    template <bool Signed = kSigned>
    static __device__ __forceinline__ C ghost(uint32_t code, C nb, C eP) {   // (code: the face's two bits)
        if (code == 0u) return nb;
        return Signed && code == 2u ? -eP : eP;
    }
    static __device__ __forceinline__ C zero_value(const C (&ih)[3], uint32_t f, C eP, C v) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if ((f >> (4 * a)) & 2u) v = fma((C)2 * ih[a], eP, v);
            if ((f >> (4 * a)) & 8u) v = fma((C)2 * ih[a], eP, v);
        }
        return v;
    }
    // one cell (any axes): e the array read, off its offset from the first e array.  The loads do
    // not wait for the code: a neighbour that the code rules out is read from valid memory and dropped.
    __device__ __forceinline__ C A1(const Slab<C>& s, const C* e, int off, uint32_t f, int c, C eP) const {
        const int own = s.own, P = s.P, last = own - 1;
        C acc = (C)0;
        const C lo_ = c >= P ? e[c - P] : s.prev[off + c], hi_ = c + P < own ? e[c + P] : s.next[off + c + P - own];
        const int sh = 4 * s.slow;
        if (s.x) {
            const C lo = e[max(c - 1, 0)], hi = e[min(c + 1, last)];
            acc = (ghost(f & 3u, lo, eP) + ghost((f >> 2) & 3u, hi, eP)) * s.ih[0];
        }
        if (s.y) {
            const C lo = e[max(c - s.nx, 0)], hi = e[min(c + s.nx, last)];
            acc = fma(ghost((f >> 4) & 3u, lo, eP) + ghost((f >> 6) & 3u, hi, eP), s.ih[1], acc);
        }
        const uint32_t fs = f >> sh;
        acc = fma(ghost(fs & 3u, lo_, eP) + ghost((fs >> 2) & 3u, hi_, eP), s.ih[s.slow], acc);
        C v = fma(s.diag, eP, -acc);
        if (!kSigned && (f & 0xaaau)) {
            const C ih[3] = {s.ih[0], s.ih[1], s.ih[2]};
            v = zero_value(ih, f, eP, v);
        }
        return v;
    }
    // four cells c .. c + 3 of a row (quads): m their values, ya / yb the rows below and above
    __device__ __forceinline__ Quad<C> A4(const Slab<C>& s, const C* e, int off, uint2 w, int c, const Quad<C>& m,
                                          const Quad<C>& ya, const Quad<C>& yb) const {
        const int own = s.own, P = s.P;
        C xl = e[max(c - 1, 0)], xr = e[min(c + 4, own - 1)];
        const Quad<C> za = c >= P ? load4(e + c - P) : load4(s.prev + off + c);
        const Quad<C> zb = c + P < own ? load4(e + c + P) : load4(s.next + off + c + P - own);
        const C ih[3] = {s.ih[0], s.ih[1], s.ih[2]}, diag = s.diag;
        // the outer x faces of the quad (a row's ends are among them) by sign, any other face and
        // solid cells in a second form: most warps hold a row's end and nothing else
        xl = ghost<true>(w.x & 3u, xl, m.v[0]);
        xr = ghost<true>((w.y >> 18) & 3u, xr, m.v[3]);
        Quad<C> o;
        if (!kSigned && !((w.x & 0x1fff1ffcu) | (w.y & 0x1ff31fffu))) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const C lo = q == 0 ? xl : m.v[q - 1], hi = q == 3 ? xr : m.v[q + 1];
                C acc = (lo + hi) * ih[0];
                acc = fma(ya.v[q] + yb.v[q], ih[1], acc);
                acc = fma(za.v[q] + zb.v[q], ih[2], acc);
                o.v[q] = fma(diag, m.v[q], -acc);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t f = code_of(w, q);
                const C eP = m.v[q];
                const C lo = q == 0 ? xl : ghost(f & 3u, m.v[q - 1], eP);
                const C hi = q == 3 ? xr : ghost((f >> 2) & 3u, m.v[q + 1], eP);
                C acc = (lo + hi) * ih[0];
                acc = fma(ghost((f >> 4) & 3u, ya.v[q], eP) + ghost((f >> 6) & 3u, yb.v[q], eP), ih[1], acc);
                acc = fma(ghost((f >> 8) & 3u, za.v[q], eP) + ghost((f >> 10) & 3u, zb.v[q], eP), ih[2], acc);
                o.v[q] = fma(diag, eP, -acc);
            }
        }
        if (!kSigned && ((w.x & 0x0aaa0aa8u) | (w.y & 0x0aa20aaau))) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t f = code_of(w, q) & (q == 0 ? 0xaa8u : (q == 3 ? 0xaa2u : 0xaaau));
                if (f) o.v[q] = zero_value(ih, f, m.v[q], o.v[q]);
            }
        }
        return o;
    }

    // the swept values of the quad c
    __device__ __forceinline__ Quad<C> sweep4(const Slab<C>& s, const C* e, int off, int c, C wiD) const {
        const uint2 w = codes4(s, c);
        const Quad<C> m = load4(e + c);
        const Quad<C> ya = load4(e + max(c - s.nx, 0)), yb = load4(e + min(c + s.nx, s.own - 4));
        const Quad<C> r = rhs4(s, c);
        const Quad<C> A = A4(s, e, off, w, c, m, ya, yb);
        Quad<C> v;
#pragma unroll
        for (int q = 0; q < 4; ++q) v.v[q] = fma(wiD, r.v[q] - A.v[q], m.v[q]);
        if ((w.x | w.y) & 0x10001000u) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (is_solid(code_of(w, q))) v.v[q] = (C)0;
        }
        return v;
    }
    // sweeps first .. last - 1 of one side of a level
    __device__ __forceinline__ void sweeps(int l, int side, int first, int last, unsigned& cur) const {
        const Slab<C>& s = tab[l];
        for (int it = first; it < last; ++it) {
            const int off = ((cur >> l) & 1u) ? s.flip : 0;
            const C* const e = sm + s.e0 + off;
            C* const o = sm + s.e0 + (s.flip - off);
            const C wiD = weight(s, side, it) * s.iD;
            if (s.quads) {
                for (int c = 4 * tid; c < s.own; c += 4 * T) store4(o + c, sweep4(s, e, off, c, wiD));
            } else {
                for (int c = tid; c < s.own; c += T) {
                    const uint32_t f = code(s, c);
                    const C r = rhs(s, c), eP = e[c];
                    const C v = fma(wiD, r - A1(s, e, off, f, c, eP), eP);
                    o[c] = is_solid(f) ? (C)0 : v;
                }
            }
            cur ^= 1u << l;
            barrier(s.all);
        }
    }

    // Residual and restriction.  Where both children planes of a coarse plane are this block's
    // (joined), the coarse r and its first sweep from e = 0.  Otherwise the sums over the in-plane
    // children, one per fine plane, into the coarse plane's block: even planes into its r, odd ones
    // into its second e array (free until its second sweep); the coarse level adds the two.
    __device__ __forceinline__ C* partial(int l, int kf) const {   // where fine plane kf's sums go
        const ClusterLevel<C>& Lc = k.lv[l + 1];
        const int K = kf >> 1;
        C* const a = sm + ((kf & 1) ? Lc.e1 : Lc.r);
        if (!dealt(l + 1)) return at(a, 0) + K * Lc.P;
        const int owner = K / Lc.m;
        return at(a, owner) + (K - owner * Lc.m) * Lc.P;
    }
    // r - A e of the 2 x 4 fine cells from c on, summed in fours
    __device__ __forceinline__ void residual8(const Slab<C>& s, const C* e, int off, int c, C& s0, C& s1) const {
        const int nx = s.nx, own = s.own;
        const uint2 wa = codes4(s, c), wb = codes4(s, c + nx);
        const Quad<C> a = load4(e + c), b = load4(e + c + nx);
        const Quad<C> lo = load4(e + max(c - nx, 0)), hi = load4(e + min(c + 2 * nx, own - 4));
        const Quad<C> ra = rhs4(s, c), rb = rhs4(s, c + nx);
        Quad<C> A = A4(s, e, off, wa, c, a, lo, b), B = A4(s, e, off, wb, c + nx, b, a, hi);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            A.v[t] = ra.v[t] - A.v[t];
            B.v[t] = rb.v[t] - B.v[t];
        }
        if ((wa.x | wa.y | wb.x | wb.y) & 0x10001000u) {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (is_solid(code_of(wa, t))) A.v[t] = (C)0;
                if (is_solid(code_of(wb, t))) B.v[t] = (C)0;
            }
        }
        s0 = (A.v[0] + A.v[1]) + (B.v[0] + B.v[1]);
        s1 = (A.v[2] + A.v[3]) + (B.v[2] + B.v[3]);
    }
    __device__ __forceinline__ C children(int l) const {   // 1 / the children of a cell of level l + 1
        const ClusterLevel<C>& L = k.lv[l];
        return (L.act[0] ? (C)0.5 : (C)1) * (L.act[1] ? (C)0.5 : (C)1) * (L.act[2] ? (C)0.5 : (C)1);
    }
    // level l + 1 at its cell c of this block: r and the first sweep
    __device__ __forceinline__ void first_at(const Slab<C>& t, C wiD, int c, C r) const {
        sm[t.r + c] = r;
        sm[t.e0 + c] = is_solid(codes()[t.f + c]) ? (C)0 : wiD * r;
    }
    __device__ __forceinline__ void restrict_to_next(int l, unsigned cur) const {
        const Slab<C>& s = tab[l];
        const Slab<C>& t = tab[l + 1];
        const int off = ((cur >> l) & 1u) ? s.flip : 0, P = s.P, Pc = t.P;
        const C* const e = sm + s.e0 + off;
        const bool joined = s.joined;
        const int np = joined ? s.np >> 1 : s.np;
        const C inv = children(l), wiD = joined ? weight(t, 0, 0) * t.iD : (C)0;
        if (s.quads) {   // two coarse cells per thread
            const int nx = s.nx, H = nx >> 2, cnx = nx >> 1, per = Pc >> 1;
            if (tid >= np * per) return;
            const float iper = 1.0f / (float)per, iH = 1.0f / (float)H;
            for (int q = tid; q < np * per; q += T) {
                const int kk = small_div(q, iper), w = q - kk * per;
                const int J = small_div(w, iH), I = w - J * H;
                const int in = 2 * J * nx + 4 * I, cc = J * cnx + 2 * I;
                C s0, s1;
                if (joined) {
                    C a0, a1;
                    residual8(s, e, off, 2 * kk * P + in, s0, s1);
                    residual8(s, e, off, (2 * kk + 1) * P + in, a0, a1);
                    first_at(t, wiD, kk * Pc + cc, (s0 + a0) * inv);
                    first_at(t, wiD, kk * Pc + cc + 1, (s1 + a1) * inv);
                } else {
                    residual8(s, e, off, kk * P + in, s0, s1);
                    C* const dst = partial(l, s.k0 + kk) + cc;
                    dst[0] = s0;
                    dst[1] = s1;
                }
            }
            return;
        }
        const int nx = s.nx, fx = s.x ? 2 : 1, fy = s.y ? 2 : 1, cnx = nx / fx;
        if (tid >= np * Pc) return;
        const float iPc = 1.0f / (float)Pc, icnx = 1.0f / (float)cnx;
        for (int q = tid; q < np * Pc; q += T) {
            const int kk = small_div(q, iPc), cc = q - kk * Pc;
            const int J = small_div(cc, icnx), I = cc - J * cnx;
            const int nz = joined ? 2 : 1;
            C sums[2] = {(C)0, (C)0};
            for (int z = 0; z < nz; ++z) {
                const int c0 = (nz * kk + z) * P + J * fy * nx + I * fx;
                C sum = (C)0;
                for (int dy = 0; dy < fy; ++dy)
                    for (int dx = 0; dx < fx; ++dx) {
                        const int c = c0 + dy * nx + dx;
                        const uint32_t f = code(s, c);
                        if (!is_solid(f)) sum += rhs(s, c) - A1(s, e, off, f, c, e[c]);
                    }
                if (z == 0) sums[0] = sum;
                else sums[1] = sum;
            }
            if (joined) first_at(t, wiD, q, (sums[0] + sums[1]) * inv);
            else partial(l, s.k0 + kk)[cc] = sums[0];
        }
    }
    // level l > 0 from the two partial sums
    __device__ __forceinline__ void first_sweep(int l) const {
        const Slab<C>& s = tab[l];
        const C inv = children(l - 1), wiD = weight(s, 0, 0) * s.iD;
        for (int c = tid; c < s.own; c += T) first_at(s, wiD, c, (sm[s.r + c] + sm[s.e0 + s.flip + c]) * inv);
    }

    // e += the trilinear interpolation of level l + 1's correction (Eq. prolongation, see prolong_at)
    __device__ __forceinline__ void prolong(int l, unsigned cur) const {
        const Slab<C>& s = tab[l];
        const Slab<C>& t = tab[l + 1];
        const ClusterLevel<C>& Lc = k.lv[l + 1];
        const int np = s.np, kf0 = s.k0, Pc = t.P;
        const int off = ((cur >> l) & 1u) ? s.flip : 0;
        C* const ef = sm + s.e0 + off;
        C* const src = sm + t.e0 + (((cur >> (l + 1)) & 1u) ? t.flip : 0);
        const C* ec = src;
        int Kb = 0;   // the plane of level l + 1 that ec starts with
        if (s.all) {
            // the coarse planes around this slab, copied from their blocks into the array that the
            // next sweep writes
            C* const buf = sm + s.e0 + (s.flip - off);
            if (np > 0) {
                const int klast = kf0 + np - 1;
                Kb = max((kf0 >> 1) - ((kf0 & 1) ? 0 : 1), 0);
                const int Ke = min((klast >> 1) + ((klast & 1) ? 1 : 0), Lc.ns - 1), m = Lc.m;
                const int total = (Ke - Kb + 1) * Pc;
                const float iPc = 1.0f / (float)Pc;
                auto from = [&](int q) -> const C* {   // coarse cell q counted from plane Kb
                    const int kk = small_div(q, iPc), K = Kb + kk;
                    if (!t.all) return at(src, 0) + Kb * Pc + q;
                    const int owner = K / m;
                    return at(src, owner) + (K - owner * m) * Pc + (q - kk * Pc);
                };
                if (Pc % 4 == 0) {
                    for (int q = 4 * tid; q < total; q += 4 * T) store4(buf + q, load4(from(q)));
                } else {
                    for (int q = tid; q < total; q += T) buf[q] = *from(q);
                }
            }
            ec = buf;
            __syncthreads();
        }
        const uint16_t* const cnbf = Lc.nbf;
        if (s.quads) {
            // four x cells per thread: the coarse cells under them and one on either side, the four
            // coarse rows (parent and neighbour along y and z) combined first
            const int H = s.nx >> 2, per = s.P >> 2, cnx = Lc.n[0], cny = Lc.n[1], ns = Lc.ns;
            const uint32_t dir = Lc.dir;
            const float iper = 1.0f / (float)per, iH = 1.0f / (float)H;
            for (int q = tid; q < np * per; q += T) {
                const int kk = small_div(q, iper), w = q - kk * per;
                const int j = small_div(w, iH), I = w - j * H, kf = kf0 + kk;
                const int c = 4 * q, I0 = 2 * I;   // (a slab's quads are consecutive)
                const int K = kf >> 1, qK = K + ((kf & 1) ? 1 : -1);
                const int J = j >> 1, qJ = J + ((j & 1) ? 1 : -1);
                const bool outK = qK < 0 || qK >= ns, outJ = qJ < 0 || qJ >= cny;
                const bool outl = I == 0, outr = I == H - 1;
                const int Ks = outK ? K : qK, Js = outJ ? J : qJ;
                const int xl = outl ? 0 : I0 - 1, xr = outr ? I0 + 1 : I0 + 2;
                // a ghost across a zero-value face of the coarse level: signed by the cells' codes
                const bool sg = dir && ((outl && (dir & 1u)) || (outr && (dir & 2u)) || (outJ && (dir & (qJ < 0 ? 4u : 8u))) ||
                                        (outK && (dir & (qK < 0 ? 16u : 32u))));
                C v0 = (C)0, v1 = (C)0, vl = (C)0, vr = (C)0;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int KK = (h & 2) ? Ks : K, JJ = (h & 1) ? Js : J;
                    const C wt = (h == 0 ? (C)0.5625 : (h == 3 ? (C)0.0625 : (C)0.1875));
                    const C* const row = ec + (KK - Kb) * Pc + JJ * cnx;
                    C a, b, l0 = row[xl], r0 = row[xr];
                    load2(row + I0, a, b);
                    if (sg) {
                        const uint16_t* const fc = cnbf + KK * Pc + JJ * cnx;
                        const uint32_t my = (h & 1) && outJ ? (qJ < 0 ? 0x20u : 0x80u) : 0u;
                        const uint32_t mz = (h & 2) && outK ? (qK < 0 ? 0x200u : 0x800u) : 0u;
                        const uint32_t fa = __ldg(fc + I0), fb = __ldg(fc + I0 + 1);
                        const uint32_t fl = outl ? fa : (uint32_t)__ldg(fc + xl);
                        const uint32_t fr = outr ? fb : (uint32_t)__ldg(fc + xr);
                        auto neg = [&](uint32_t f, uint32_t mx) {
                            return (((f & my) != 0u) != ((f & mz) != 0u)) != ((f & mx) != 0u);
                        };
                        if (neg(fa, 0u)) a = -a;
                        if (neg(fb, 0u)) b = -b;
                        if (neg(fl, outl ? 0x2u : 0u)) l0 = -l0;
                        if (neg(fr, outr ? 0x8u : 0u)) r0 = -r0;
                    }
                    v0 = fma(wt, a, v0);
                    v1 = fma(wt, b, v1);
                    vl = fma(wt, l0, vl);
                    vr = fma(wt, r0, vr);
                }
                const uint2 fw = codes4(s, c);
                Quad<C> m = load4(ef + c);
                const C add[4] = {fma((C)0.25, vl, (C)0.75 * v0), fma((C)0.25, v1, (C)0.75 * v0),
                                  fma((C)0.25, v0, (C)0.75 * v1), fma((C)0.25, vr, (C)0.75 * v1)};
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    if (!is_solid(code_of(fw, h))) m.v[h] += add[h];
                store4(ef + c, m);
            }
        } else {   // cell by cell
            const int nx = s.nx, rows = s.P / nx, slow = s.slow;
            const float inx = 1.0f / (float)nx, irows = 1.0f / (float)rows;
            const ClusterLevel<C>& L = k.lv[l];
            const int fa[3] = {L.act[0], L.act[1], L.act[2]}, cn[3] = {Lc.n[0], Lc.n[1], Lc.n[2]};
            const C* const shifted = ec - (ptrdiff_t)Kb * Pc;
            for (int q = tid; q < s.own; q += T) {
                if (is_solid(code(s, q))) continue;
                const int row = small_div(q, inx), i = q - row * nx;
                const int kk = small_div(row, irows), j = row - kk * rows, kf = kf0 + kk;
                ef[q] += prolong_at<C>(fa, cn, slow == 0 ? kf : i, slow == 1 ? kf : j, slow == 2 ? kf : 0,
                                       [&](int x) { return shifted[x]; }, [&](int x) { return (uint32_t)__ldg(cnbf + x); });
            }
        }
    }

    // e = A^-1 r on the coarsest level: a warp takes up to four rows of the dense inverse at
    // once, the result in block 0's e (in e_out where the coarsest level is the cluster's only one)
    __device__ __forceinline__ void dense(int warp, int warps) const {
        const ClusterLevel<C>& L = k.lv[k.nl - 1];
        const int N = L.ns * L.P;
        const bool only = k.nl == 1;
        C* const x = sm + k.x;
        if (only) {
            for (int c = tid; c < N; c += T) x[c] = to_c<C>(ldg(k.r_in + c));
        } else {
            const C inv = children(k.nl - 2);
            const C* const a = at(sm + L.r, 0);
            const C* const b = at(sm + L.e1, 0);
            for (int c = tid; c < N; c += T) x[c] = (a[c] + b[c]) * inv;
        }
        __syncthreads();
        C* const out = only ? nullptr : at(sm + L.e0, 0);
        if (N > 2 * warps) rows_of<4>(N, x, out, warp, warps);
        else rows_of<1>(N, x, out, warp, warps);
    }
    template <int R>
    __device__ __forceinline__ void rows_of(int N, const C* x, C* out, int warp, int warps) const {
        const int lane = tid & 31;
        const C* const Ai = inverse(N);
        for (int row = warp; row < N; row += R * warps) {
            const C* a[R];
            C acc[R];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                a[q] = Ai + (size_t)min(row + q * warps, N - 1) * N;
                acc[q] = (C)0;
            }
            if (N % 4 == 0) {
#pragma unroll 2
                for (int col = 4 * lane; col < N; col += 128) {
                    const Quad<C> xv = load4(x + col);
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        const Quad<C> av = load4(a[q] + col);
#pragma unroll
                        for (int h = 0; h < 4; ++h) acc[q] = fma(av.v[h], xv.v[h], acc[q]);
                    }
                }
            } else {
                for (int col = lane; col < N; col += 32)
#pragma unroll
                    for (int q = 0; q < R; ++q) acc[q] = fma(__ldg(a[q] + col), x[col], acc[q]);
            }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                for (int off = 16; off > 0; off >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
                const int to = row + q * warps;
                if (lane == 0 && to < N) {
                    if (out) out[to] = acc[q];
                    else k.e_out[to] = from_c<TI, C>(acc[q]);
                }
            }
        }
    }
    __device__ __forceinline__ const C* inverse(int N) const {   // (the FP32 copy follows the FP64 inverse)
        return reinterpret_cast<const C*>(sizeof(C) == 8 ? k.Ainv : k.Ainv + (size_t)N * N);
    }

    // what no earlier launch writes, before waiting for it: the levels' table, their codes into
    // shared memory, and the dense inverse named to L2
    __device__ __forceinline__ void prologue() const {
        const int last = k.nl - 1;
        if (tid < k.nl) form_slab(tid);
        __syncthreads();
        if (last > 0)
            for (int l = 0; l < k.nl; ++l) {
                const Slab<C>& s = tab[l];
                if (s.f < 0) continue;
                uint16_t* const F = reinterpret_cast<uint16_t*>(sm) + s.f;
                const uint16_t* const src = s.nbf;
                const int own = s.own;
                if (s.P % 4 == 0)
#pragma unroll 4
                    for (int c = 4 * tid; c < own; c += 4 * T)
                        *reinterpret_cast<uint2*>(F + c) = __ldg(reinterpret_cast<const uint2*>(src + c));
                else
                    for (int c = tid; c < own; c += T) F[c] = __ldg(src + c);
            }
        if (k.dense_all || last == 0) {
            const int N = k.lv[last].ns * k.lv[last].P, line = 128 / (int)sizeof(C);
            const C* const a = inverse(N);
            for (int q = (rank * T + tid) * line; q < N * N; q += k.S * T * line)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a + q));
        }
    }

    __device__ __forceinline__ void run() const {
        const int last = k.nl - 1;
        if (last == 0) {
            dense(rank * (T >> 5) + (tid >> 5), k.S * (T >> 5));
            return;
        }
        unsigned cur = 0u;   // bit l: the array that holds level l's correction
        {   // the finest level's r and its first sweep
            __syncthreads();   // (the codes)
            const Slab<C>& s = tab[0];
            const C wiD = weight(s, 0, 0) * s.iD;
            const TI* const rg = k.r_in + s.base;
            const int own = s.own, ro = s.r;
            C* const E0 = sm + s.e0;
            if (s.P % 4 == 0) {
#pragma unroll 2
                for (int c = 4 * tid; c < own; c += 4 * T) {
                    Quad<C> r = load4(rg + c);
                    const uint2 w = codes4(s, c);
                    if (ro >= 0) store4(sm + ro + c, r);
#pragma unroll
                    for (int q = 0; q < 4; ++q) r.v[q] = is_solid(code_of(w, q)) ? (C)0 : wiD * r.v[q];
                    store4(E0 + c, r);
                }
            } else {
                for (int c = tid; c < own; c += T) {
                    const C r = to_c<C>(ldg(rg + c));
                    if (ro >= 0) sm[ro + c] = r;
                    E0[c] = is_solid(code(s, c)) ? (C)0 : wiD * r;
                }
            }
        }
        barrier(dealt(0));
        for (int l = 0; l < last; ++l) {
            if (!dealt(l) && rank != 0) break;
            if (l > 0 && !tab[l - 1].joined) {
                first_sweep(l);
                barrier(dealt(l));
            }
            sweeps(l, 0, 1, k.pre, cur);
            restrict_to_next(l, cur);
            barrier(dealt(l));
        }
        if (k.dense_all) {
            if (k.lm < last) cluster_barrier();   // block 0's restriction, before the others read it
            dense(rank * (T >> 5) + (tid >> 5), k.S * (T >> 5));
            cluster_barrier();
        } else if (rank == 0) {
            dense(tid >> 5, T >> 5);
            __syncthreads();
        }
        // (every block counts the sweeps of block 0's levels the same way)
        if (rank != 0)
            for (int l = k.lm; l < last; ++l)
                if (((k.pre - 1 + k.post) & 1) != 0) cur ^= 1u << l;
        for (int l = last - 1; l >= 0; --l) {
            if (l == k.lm - 1 && !(k.dense_all && k.lm == last)) cluster_barrier();   // block 0's correction is complete
            if (!dealt(l) && rank != 0) continue;
            prolong(l, cur);
            barrier(dealt(l));
            sweeps(l, 1, 0, k.post, cur);
        }
        {
            const Slab<C>& s = tab[0];
            const int own = s.own;
            const C* const v = sm + s.e0 + ((cur & 1u) ? s.flip : 0);
            TI* const out = k.e_out + s.base;
            if (k.p) {
                double* const p = k.p + s.base;   // (pairs where the corrections are not FP64: pp_load)
                for (int c = tid; c < own; c += T) {
                    if constexpr (sizeof(C) == 8) {
                        p[c] += v[c];
                    } else {
                        float2* const q = reinterpret_cast<float2*>(p) + c;
                        *q = pp_plus(*q, v[c]);
                    }
                }
            } else if (s.P % 4 == 0)
                for (int c = 4 * tid; c < own; c += 4 * T) store4(out + c, load4(v + c));
            else
                for (int c = tid; c < own; c += T) out[c] = from_c<TI, C>(v[c]);
        }
    }
};

extern __shared__ __align__(16) unsigned char g_coarse_smem[];

__device__ __forceinline__ int block_rank(int S) { return S > 1 ? (int)(blockIdx.x % (unsigned)S) : 0; }

template <class TI>
__global__ void __launch_bounds__(kCtaThreads, 1) k_coarse(const __grid_constant__ CoarseK<TI> k) {
    __shared__ Slab<typename Acc<TI>::type> tab[FVM_MAX_LEVELS];
    const Body<TI> b(k, g_coarse_smem, tab, block_rank(k.S));
    b.prologue();
    pdl_enter();
    b.run();
}

// a batch: one cluster per case
template <class TI>
__global__ void __launch_bounds__(kCtaThreads, 1) k_coarse_many(const CoarseK<TI>* __restrict__ ks, int S) {
    __shared__ __align__(16) unsigned char buf[sizeof(CoarseK<TI>)];
    const uint32_t* src = reinterpret_cast<const uint32_t*>(ks + blockIdx.x / (unsigned)S);
    for (int q = threadIdx.x; q < (int)(sizeof(CoarseK<TI>) / 4); q += blockDim.x)
        reinterpret_cast<uint32_t*>(buf)[q] = __ldg(src + q);
    __syncthreads();
    const CoarseK<TI>& k = *reinterpret_cast<const CoarseK<TI>*>(buf);
    __shared__ Slab<typename Acc<TI>::type> tab[FVM_MAX_LEVELS];
    const Body<TI> b(k, g_coarse_smem, tab, block_rank(S));
    b.prologue();
    // (the next kernel starts when this one ends: its blocks, let in early, kept the last clusters from
    // finding their blocks' shared memory, 250 us a V-cycle with 64 cases; eight cases lose 0.5 %)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (k.st->active == 0) return;   // a converged case: its whole cluster leaves
    b.run();
}

cudaLaunchConfig_t cluster_config(cudaLaunchAttribute* attr, unsigned blocks, int S, size_t smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kCtaThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    unsigned n = 0;
    if (S > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)S;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (pdl_enabled() && s) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cfg;
}

// the kernel may be launched as clusters of S blocks with this much shared memory (its limits
// are raised; a launch that the device cannot hold is not issued)
cudaError_t prepare_kernel(const void* fn, int S, size_t smem) {
    cudaError_t e = raise_smem_limit(fn, smem);
    if (e != cudaSuccess) return e;
    if (S > 8 && (e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) {
        cudaGetLastError();
        return e;
    }
    if (S > 1) {
        cudaLaunchAttribute attr[2];
        const cudaLaunchConfig_t cfg = cluster_config(attr, (unsigned)S, S, smem, nullptr);
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
        if (e != cudaSuccess || n < 1) {
            cudaGetLastError();
            return cudaErrorInvalidConfiguration;
        }
    }
    return cudaSuccess;
}

template <class TI>
cudaError_t coarse_many(const void* tab, const BatchMap& m, unsigned nblk, dim3, size_t smem, const BatchCtl*,
                        cudaStream_t s) {
    const void* fn = (const void*)k_coarse_many<TI>;
    const int S = m.total / m.n;   // every case's grid is one cluster of the same size
    if (nblk == 0) return prepare_kernel(fn, S, smem);
    if (!smem_limit_covers(fn, smem)) return cudaErrorInvalidConfiguration;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(attr, nblk, S, smem, s);
    return cudaLaunchKernelEx(&cfg, k_coarse_many<TI>, (const CoarseK<TI>*)tab, S);
}

template <class TI>
CoarseK<TI> functor(const CoarsePlan& pl, const void* r_in, void* e_out, double* p, const double* Ainv,
                    const SolveState* st) {
    using C = typename Acc<TI>::type;
    CoarseK<TI> k;
    memset(&k, 0, sizeof(k));
    k.S = pl.S;
    k.nl = pl.nl;
    k.lm = pl.lm;
    k.pre = pl.pre;
    k.post = pl.post;
    k.cheb = pl.cheb;
    k.dense_all = pl.dense_all;
    k.x = pl.x;
    for (int l = 0; l < pl.nl; ++l) {
        const CoarsePlan::Level& p = pl.lv[l];
        const LevelDev& v = p.dev;
        ClusterLevel<C>& L = k.lv[l];
        for (int a = 0; a < 3; ++a) {
            L.n[a] = v.n[a];
            L.act[a] = v.active[a] != 0;
            L.ih[a] = sizeof(C) == 8 ? (C)v.ih2a[a] : (C)v.ih2af[a];
        }
        L.slow = p.slow;
        L.P = p.P;
        L.ns = p.ns;
        L.m = p.m;
        L.e0 = p.e0;
        L.e1 = p.e1;
        L.r = p.r;
        L.f = p.f;
        L.dir = p.dir;
        L.diag = sizeof(C) == 8 ? (C)v.diag : (C)v.diagf;
        L.iD = sizeof(C) == 8 ? (C)v.inv_D : (C)v.inv_Df;
        L.wJ = sizeof(C) == 8 ? (C)v.wJ : (C)v.wJf;
        L.nbf = v.nbf;
    }
    for (int side = 0; side < 2; ++side)
        for (int i = 0; i < kMaxChebSweeps; ++i) k.w[side][i] = (C)pl.w[side][i];
    k.r_in = (const TI*)r_in;
    k.e_out = (TI*)e_out;
    k.p = p;
    k.Ainv = Ainv;
    k.st = st;
    return k;
}

template <class TI>
cudaError_t launch(const CoarsePlan& pl, const void* r_in, void* e_out, double* p, const double* Ainv,
                   const SolveState* st, cudaStream_t s) {
    const CoarseK<TI> k = functor<TI>(pl, r_in, e_out, p, Ainv, st);
    if (record_launch(k, dim3((unsigned)pl.S), dim3(kCtaThreads), pl.smem, &coarse_many<TI>)) return cudaSuccess;
    const void* fn = (const void*)k_coarse<TI>;
    if (!smem_limit_covers(fn, pl.smem)) return cudaErrorInvalidConfiguration;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(attr, (unsigned)pl.S, pl.S, pl.smem, s);
    return cudaLaunchKernelEx(&cfg, k_coarse<TI>, k);
}

}  // namespace

// Cells from which a level is dealt out over the cluster's blocks, and unknowns from which the
// dense solve is: below them block 0 alone is quicker than a cluster barrier per phase (a sweep
// of 64 to 2048 FP32 cells on one block 0.5 us, dealt out 0.9 us; FP64 arithmetic runs at 1/64 of
// the FP32 rate, two lanes a clock and SM).
static int deal_from(int inner) { return inner == FVM_FP64 ? 192 : 2048; }
static int dense_all_from(int inner) { return inner == FVM_FP64 ? 64 : 160; }
// The finest level a cluster takes, in cells per block: up to 65,536 cells in FP32 and BF16, 8192
// in FP64 on 16 blocks.  Beyond, the grid-wide launches spread a sweep over 152 SMs and win: ten
// steps of the 256 x 64 x 64 FP32 channel took 8.91 ms with its 2048-cell level as the finest in
// the cluster, 8.54 ms with the 16,384-cell level, 8.73 ms with the 131,072-cell level; four of
// the FP64 channel 26.8, 27.1 (16,384 cells) and 30.7 ms; four of the 512 x 256 x 128 BF16 room
// 54.4 ms with 32,768 cells, 55.8 ms with 262,144.
static int64_t cells_per_block(int inner, int S) {
    if (S == 1) return inner == FVM_FP64 ? 512 : 8192;
    return inner == FVM_FP64 ? 512 : 4096;
}
constexpr size_t kSmemBudget = 222 * 1024;   // (227 KB less the static arrays)

bool coarse_plan_from(const std::vector<LevelDev>& levels, const std::vector<uint32_t>& dir, int inner, int S, int lc,
                      CoarsePlan& pl) {
    memset((void*)&pl, 0, sizeof(pl));
    pl.S = S;
    pl.lc = lc;
    pl.nl = (int)levels.size() - lc;
    const size_t cs = inner == FVM_FP64 ? 8 : 4;
    for (int top_global = 0; top_global < 2; ++top_global) {
        size_t q = 0, codes = 0;
        pl.lm = 0;
        for (int l = 0; l < pl.nl; ++l) {
            const LevelDev& v = levels[lc + l];
            CoarsePlan::Level& p = pl.lv[l];
            p.dev = v;
            p.dir = dir[lc + l];
            p.slow = v.active[2] ? 2 : (v.active[1] ? 1 : 0);
            p.ns = v.n[p.slow];
            p.P = (int)(v.N / p.ns);
            const bool deal = S > 1 && l + 1 < pl.nl && v.N >= deal_from(inner);   // (never the coarsest)
            p.m = deal ? (p.ns + S - 1) / S : p.ns;
            if (deal) pl.lm = l + 1;
            const size_t own = pl.nl > 1 ? (size_t)p.m * p.P : 0;   // (the dense solve alone needs only x)
            // the coarse planes around a slab are copied into the e array a sweep would write next
            const size_t coarse_planes = l + 1 < pl.nl ? (size_t)(p.m / 2 + 2) * (levels[lc + l + 1].N / (p.ns / 2)) : 0;
            const size_t ecells = ((own > coarse_planes ? own : coarse_planes) + 3) / 4 * 4;
            p.e0 = (int)q;
            q += ecells;
            p.e1 = (int)q;
            q += ecells;
            if (l == 0 && top_global) {
                p.r = -1;
                p.f = -1;
            } else {
                p.r = (int)q;
                q += (own + 3) / 4 * 4;
                codes += (own + 3) / 4 * 4;
            }
        }
        pl.x = (int)q;
        q += ((size_t)levels.back().N + 3) / 4 * 4;
        size_t u = q * (cs / 2);
        for (int l = 0; l < pl.nl; ++l)
            if (pl.lv[l].r >= 0) {
                pl.lv[l].f = (int)u;
                u += ((size_t)pl.lv[l].m * pl.lv[l].P + 3) / 4 * 4;
            }
        pl.smem = q * cs + codes * 2 + 16;
        pl.dense_all = pl.S > 1 && pl.lm > 0 && levels.back().N >= dense_all_from(inner) ? 1 : 0;
        if (pl.smem <= kSmemBudget) return true;
    }
    return false;
}

bool coarse_plan(const std::vector<LevelDev>& levels, const std::vector<uint32_t>& dir, int inner, int S, bool exact,
                 int first, CoarsePlan& pl) {
    // level 0 itself: where its cells go through the four-cell forms as much as any level, else half of
    // that in FP64 and a quarter in FP32 and BF16.  Ten steps of six V-cycles, level 0 in the cluster
    // against in launches: FP64 plane of 4096 cells 3.88 / 4.10 ms, of 8192 4.28 / 4.28, FP64 box of 8192
    // 5.06 / 5.13; FP32 boxes of 8192 cells 2.50 / 2.75, 32,768 2.84 / 3.13, 65,536 3.19 / 3.29, plane of
    // 8192 2.73 / 2.93, of 16,384 3.09 / 3.25, of 32,768 3.41 / 3.30
    if (first == 0) {
        const LevelDev& v = levels[0];
        const bool quads = v.active[0] && v.active[1] && v.active[2] && v.n[0] % 4 == 0;
        if (!quads && v.N > cells_per_block(inner, S) * S / (inner == FVM_FP64 ? 2 : 4)) first = 1;
    }
    for (int lc = first; lc < (int)levels.size(); ++lc) {
        if (levels[lc].N > cells_per_block(inner, S) * S && lc + 1 < (int)levels.size()) continue;
        if (!coarse_plan_from(levels, dir, inner, S, lc, pl)) continue;
        if (exact || S == 1 || pl.lm > 0 || pl.nl == 1) return true;
        return coarse_plan_from(levels, dir, inner, 1, lc, pl) || coarse_plan_from(levels, dir, inner, S, lc, pl);
    }
    return false;
}

// (the results are those of any number of blocks from the same finest level: only who works on a
// cell changes, not its arithmetic)
int coarse_cluster_for(int cases) {
    for (int S : {16, 8, 4, 2})
        if (cases * S <= (S == 16 ? 112 : 144)) return S;
    return 1;
}

cudaError_t prepare_coarse(int inner, const CoarsePlan& pl) {
    const void* fn = inner == FVM_FP64   ? (const void*)k_coarse<double>
                     : inner == FVM_FP32 ? (const void*)k_coarse<float>
                                         : (const void*)k_coarse<__nv_bfloat16>;
    return prepare_kernel(fn, pl.S, pl.smem);
}

cudaError_t prepare_coarse_many(int inner, int S, size_t smem) {
    const void* fn = inner == FVM_FP64   ? (const void*)k_coarse_many<double>
                     : inner == FVM_FP32 ? (const void*)k_coarse_many<float>
                                         : (const void*)k_coarse_many<__nv_bfloat16>;
    return prepare_kernel(fn, S, smem);
}

cudaError_t launch_coarse(int inner, const CoarsePlan& pl, const void* r_in, void* e_out, double* p,
                          const double* Ainv, const SolveState* st, cudaStream_t s) {
    if (inner == FVM_FP64) return launch<double>(pl, r_in, e_out, p, Ainv, st, s);
    if (inner == FVM_FP32) return launch<float>(pl, r_in, e_out, p, Ainv, st, s);
    return launch<__nv_bfloat16>(pl, r_in, e_out, p, Ainv, st, s);
}
