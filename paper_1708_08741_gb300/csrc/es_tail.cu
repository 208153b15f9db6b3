// es_tail.cu -- the coarse part of the V-cycle in one launch (a4; Sec. 5.3).
//
// Below about 64^3 cells a level's half sweep is a few microseconds of
// launch, cache latency and drain around well under a microsecond of work,
// and a V-cycle makes up to a hundred of them; the coarsest level, in one
// block, is bound by that block's SM (in FP64 by its FP64 pipe: 0.39 ms for
// 32 sweeps of 16^3 cells).  k_tail runs the levels l0 .. L-1 of the V-cycle,
// from the right-hand side of level l0 to its correction, as one thread-block
// cluster of up to 16 blocks: the levels' e, right-hand sides and stencil
// codes live in the blocks' shared memory, a block owns a slab of z planes of
// every level and reads the planes next to it through distributed shared
// memory, and cluster barriers separate the half sweeps instead of launches.
// The arithmetic is the kernels' of es_solver.cu; in FP32 with the same
// operations in the same order, so that a reduced-form solve gives the bits of
// the levels launched one by one (TailLevel::how).  In FP64 every cell
// multiplies by the tabulated inverse of its diagonal, as k_smooth_d does.
//
// Layout in shared memory: per level the two colours apart, a row holding the
// compact places x / 2 of its cells padded to a multiple of four, so that a
// thread moves spans of four places with 16-byte accesses and a half sweep
// streams without bank conflicts.  The stencil codes (one 16-bit word a cell)
// are formed once a mapping by k_tail_codes, in the blocks' own layout, and
// come in as one bulk copy.
//
// What bounds it: a half sweep is one cluster barrier (480 cycles with its
// release fence, whatever the cluster's size), one distributed-shared-memory
// read (264 cycles) and the arithmetic (FP64: four 64-cycle operations in a
// row, and on 32^3 the FP64 pipe: six or seven instructions a warp at 17
// cycles each).  Measured per half sweep, 16 blocks: FP32 0.18 us (8^3) and 0.42
// (16^3, one block, no cluster barrier), 0.62 us (32^3), 1.6 us (48^3), 2.8 us
// (64^3); FP64 0.82 us (16^3); a launch of its own takes 1.8 us and more on such
// levels, and some 3 us next to obstacles.  V-cycle with its correction and
// residual, every level launched (when this was made) / with it: FP32 128^3
// 250 / 185 us, 96^3 208 / 139, 256^3 526 / 508, 32^3 134 / 62; FP64 32^3 202 /
// 109 us (16^3 and 8^3 in it).
// Boundary planes pushed to the neighbours with an mbarrier each, in place of
// the cluster barrier, were no faster (FP64 32^3 107 / 111 us a tail, FP32
// 96^3 150 / 164 a V-cycle): that round trip is as long.
#include <cooperative_groups.h>

#include <type_traits>

#include "es_device.cuh"

namespace es {

namespace {

namespace cg = cooperative_groups;

constexpr int kTailThreads = 512;
constexpr int kTailCluster = 16;          // most blocks of the cluster
constexpr size_t kTailSmem = 220 * 1024;  // most dynamic shared memory of a block
// A cell's code: the six faces as near_faces has them (two bits each) and in
// the top four bits 6 + (faces that raise the diagonal) - (faces that lower it);
// kTailOff: not an unknown cell.  FP32, levels that divide: kTailOdd there means
// that the diagonal formed face by face differs from diag0 plus that sum by
// rounding, kTailEven a near-boundary cell whose sum is 0 (6: interior ones).
constexpr unsigned kTailOff = 0xFFFFu, kTailInner = 6u << 12, kTailOdd = 13u, kTailEven = 14u;

struct TailShape {
    int nx, ny, nz;
    int nxh, nxp;  // compact places of a row, and padded to a multiple of 4
    int pw;        // spans of a row: nxp / kSpan
    int zs;        // planes of a block's slab
    int plane;     // places of a colour's plane: nxp ny
    int ploc;      // and of its slab
    int c, e, r;   // byte offsets in a block's shared memory: codes, e, right-hand side
    int rpi;       // rows that the block's threads cover at once, and that as
    int dz, dy;    // planes and rows
    unsigned mpw, mny, mzs;  // ceil(2^22 / d) of pw, ny, zs: t / d = (t m) >> 22 for t < 1024
};

// How the FP32 half sweeps divide by the diagonal: as k_coarse_lists (the
// coarsest level), by a tabulated inverse; as k_smooth_v, interior cells by the
// inverse of diag0 and near-boundary cells by a quotient; as k_smooth and
// k_coarse_solve, every cell by a quotient.
enum TailHow { kByTable, kNearQuotient, kQuotient };

template <class T>
struct TailLevel {
    TailShape s;
    T h2, inv_h2, diag0;
    int how;       // TailHow (FP64: by table)
    int odd;       // kTailOdd may occur
    int red_only;  // the restriction takes the red residuals only
    int pairs;     // and adds the two children of a fine row first (k_restrict_v)
    // omega != 1, FP32: omega g enters the sum (1 - omega) e + omega g unrounded
    // (else the other product does), at interior and at near-boundary cells, as
    // in the level's kernels
    int fuse_inner, fuse_near;
};

struct TailCodes {
    TailShape s[ES_MAXLEV];
    const uint8_t* st[ES_MAXLEV];
    int n, blocks, bytes;  // levels, blocks, code bytes of a block
    int per[3], pot_bc[6];
    float diag0[ES_MAXLEV];  // 0: no kTailOdd, kTailEven
    unsigned char* out;
};

template <class T>
struct TailArgs {
    TailLevel<T> lv[ES_MAXLEV];
    int n;          // levels
    const unsigned char* codes;
    int code_bytes, smem_bytes;
    const T* rhs;   // of the first level (global memory)
    T* out;         // its correction
    int half;       // 0: natural layout; else colour-split, half its cells
    int warm;       // the iterate starts from out instead of zero
    int nu1, nu2, sweeps;
    T omega;
    int solo;       // the coarsest level belongs to block 0 alone
    int* status;
};

// Places a thread moves at once: four in FP32 (16-byte accesses); one in FP64,
// whose operations cost 16 cycles a warp and 64 cycles of latency, so that
// more and shorter threads are the faster ones.
template <class T>
constexpr int kSpan = sizeof(T) == 4 ? 4 : 1;

template <class T>
struct Span {
    T v[kSpan<T>];
};

__device__ __forceinline__ Span<float> ldspan(const float* p) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    return {{q.x, q.y, q.z, q.w}};
}
__device__ __forceinline__ Span<double> ldspan(const double* p) { return {{*p}}; }
__device__ __forceinline__ void stspan(float* p, const Span<float>& s) {
    *reinterpret_cast<float4*>(p) = make_float4(s.v[0], s.v[1], s.v[2], s.v[3]);
}
__device__ __forceinline__ void stspan(double* p, const Span<double>& s) { *p = s.v[0]; }

// The codes of a span.
template <class T>
struct Codes {
    unsigned w[(kSpan<T> + 1) / 2];
    __device__ __forceinline__ explicit Codes(const unsigned short* p) {
        if constexpr (kSpan<T> == 4) {
            const uint2 q = *reinterpret_cast<const uint2*>(p);
            w[0] = q.x;
            w[1] = q.y;
        } else {
            w[0] = *p;
        }
    }
    __device__ __forceinline__ unsigned at(int k) const { return (w[k >> 1] >> (16 * (k & 1))) & 0xFFFFu; }
    __device__ __forceinline__ bool inner() const {
        if constexpr (kSpan<T> == 4)
            return w[0] == (kTailInner | (kTailInner << 16)) && w[1] == w[0];
        else
            return w[0] == kTailInner;
    }
};

// The block whose slab holds plane z.
__device__ __forceinline__ int slab_owner(const TailShape& S, int z) { return (int)(((unsigned)z * S.mzs) >> 22); }

// A level as a block sees it: its slab, the planes next to it, and the rows
// this thread takes (the span from j0 of the rows row0, row0 + rpi, ...).
template <class T>
struct Slab {
    T *e, *r;
    const unsigned short* code;
    const T *lo, *hi;  // e of the planes below and above the slab (perhaps another block's)
    int z0, nzl;       // first plane, planes
    int j0, row0, y0, lz0, nrows;

    __device__ __forceinline__ Slab(const TailShape& S, unsigned char* smem, cg::cluster_group& cl, int rank) {
        e = (T*)(smem + S.e);
        r = (T*)(smem + S.r);
        code = (const unsigned short*)(smem + S.c);
        z0 = rank * S.zs;
        nzl = min(S.zs, max(0, S.nz - z0));
        lo = hi = e;
        if (nzl > 0) {
            const int zl = z0 == 0 ? S.nz - 1 : z0 - 1, zh = z0 + nzl >= S.nz ? 0 : z0 + nzl;
            const int ol = slab_owner(S, zl), oh = slab_owner(S, zh);
            lo = cl.map_shared_rank(e, ol) + S.plane * (zl - ol * S.zs);
            hi = cl.map_shared_rank(e, oh) + S.plane * (zh - oh * S.zs);
        }
        const unsigned t = threadIdx.x;
        row0 = (int)((t * S.mpw) >> 22);
        j0 = kSpan<T> * ((int)t - row0 * S.pw);
        lz0 = (int)(((unsigned)row0 * S.mny) >> 22);
        y0 = row0 - lz0 * S.ny;
        nrows = row0 < S.rpi ? S.ny * nzl : 0;  // (threads past the last whole row take none)
    }
    // fn(row, y, lz) for this thread's rows
    template <class Fn>
    __device__ __forceinline__ void rows(const TailShape& S, Fn&& fn) const {
        int y = y0, lz = lz0;
        for (int row = row0; row < nrows; row += S.rpi) {
            fn(row, y, lz);
            y += S.dy;
            lz += S.dz;
            if (y >= S.ny) {
                y -= S.ny;
                lz++;
            }
        }
    }
};

// Where the six neighbours of a span of colour's places are, relative to the
// other colour's array of the slab (or, past its ends, of the next planes).
template <class T>
struct Around {
    int i, h, a, b;  // the span, its halo place, the rows y -+ 1
    const T *d, *f;  // the planes z -+ 1
    int O, last;     // x parity; places after the first one to the row's last
    __device__ __forceinline__ Around(const TailShape& S, const Slab<T>& s, int colour, int row, int y, int lz) {
        const int other = (1 - colour) * S.ploc, j0 = s.j0, W = kSpan<T>;
        i = row * S.nxp + j0;
        O = (colour + y + s.z0 + lz) & 1;
        last = S.nxh - 1 - j0;
        h = other + row * S.nxp + (O ? (j0 + W < S.nxh ? j0 + W : 0) : (j0 > 0 ? j0 - 1 : S.nxh - 1));
        a = other + (y == 0 ? i + S.plane - S.nxp : i - S.nxp);
        b = other + (y == S.ny - 1 ? i - S.plane + S.nxp : i + S.nxp);
        d = lz > 0 ? s.e + other + i - S.plane : s.lo + other + y * S.nxp + j0;
        f = lz + 1 < s.nzl ? s.e + other + i + S.plane : s.hi + other + y * S.nxp + j0;
        i += other;
    }
};

// The diagonal of a cell that is unknown, face by face as near_sums forms it
// (in FP32 diag0 + 1 + 1 - 1 is not always diag0 + 1).
__device__ __noinline__ float code_diag(float diag0, unsigned c) {
    float d = diag0;
#pragma unroll
    for (int f = 0; f < 6; f++) {
        const unsigned u = (c >> (2 * f)) & 3u;
        d += u == 0u ? 0.0f : (u == 1u ? 1.0f : -1.0f);
    }
    return d;
}

// A level's tables, by the top four bits of a code: inverse diagonals (0 at cells
// that are not unknown), diagonals, and in FP32 the inverses again at the cells
// that take the quotient (else 0).
template <class T>
struct Tables {
    const T *inv, *diag, *cor;
};

// The inverse diagonals of a span's cells.
template <class T>
__device__ __forceinline__ Span<T> inverses(const Tables<T>& B, const Codes<T>& cd) {
    Span<T> y;
#pragma unroll
    for (int k = 0; k < kSpan<T>; k++) y.v[k] = B.inv[cd.at(k) >> 12];
    return y;
}

// (Rare paths are calls: the kernel's time on the smallest levels is also that of
// fetching its instructions.)
__device__ __noinline__ Span<float> odd_diagonals(float diag0, Span<float> d, Codes<float> cd) {
    for (int k = 0; k < kSpan<float>; k++)
        if ((cd.at(k) >> 12) == kTailOdd) d.v[k] = code_diag(diag0, cd.at(k));
    return d;
}
__device__ __noinline__ Span<float> odd_inverses(Span<float> d, Span<float> y, Codes<float> cd) {
    for (int k = 0; k < kSpan<float>; k++)
        if ((cd.at(k) >> 12) == kTailOdd) y.v[k] = __fdiv_rn(1.0f, d.v[k]);
    return y;
}
__device__ __noinline__ Span<float> odd_quotients(float diag0, Span<float> n, Span<float> q, Codes<float> cd) {
    for (int k = 0; k < kSpan<float>; k++)
        if ((cd.at(k) >> 12) == kTailOdd) q.v[k] = n.v[k] / code_diag(diag0, cd.at(k));
    return q;
}

// n over the diagonal for a span's cells (see TailHow).  The quotient comes
// from the tabulated inverse y = RN(1 / d): q = RN(n y) is within 1.5 ulp of n / d
// (within one unless n < d), and q + (n - q d) y then rounds to n / d (P.
// Markstein, Computation of elementary functions on the IBM RISC System/6000
// processor, IBM J. Res. Dev. 34, 1990, for a q within one ulp; beyond it n / d
// would have to lie within 1.5 2^-23 ulp of a midpoint, which puts n and d
// within three ulp of 2, where it does not; 8e9 pairs tried).  So the bits of a
// division for two multiply-adds a near-boundary cell.
template <class T>
__device__ __forceinline__ Span<T> quotients(const TailLevel<T>& L, int how, int odd, const Tables<T>& B,
                                             const Span<T>& n, const Span<T>& y, const Codes<T>& cd) {
    Span<T> q;
#pragma unroll
    for (int k = 0; k < kSpan<T>; k++) q.v[k] = n.v[k] * y.v[k];
    if constexpr (sizeof(T) == 4) {
        if (how == kByTable || (how == kNearQuotient && cd.inner())) return q;
#pragma unroll
        for (int k = 0; k < kSpan<T>; k++) {
            const unsigned i = cd.at(k) >> 12;
            const T cor = how == kNearQuotient && i == 6u ? (T)0 : y.v[k];  // (as Tables::cor)
            q.v[k] = __fmaf_rn(__fmaf_rn(-q.v[k], B.diag[i], n.v[k]), cor, q.v[k]);
        }
        if (odd) q = odd_quotients(L.diag0, n, q, cd);
    }
    return q;
}

// (1 - omega) e + omega g
__device__ __forceinline__ Span<double> relaxed(const TailLevel<double>&, double omega, Span<double> e, Span<double> g,
                                                const Codes<double>&) {
    return {{(1.0 - omega) * e.v[0] + omega * g.v[0]}};
}
__device__ __noinline__ Span<float> relaxed_as(int inner, int near, float omega, Span<float> e, Span<float> g,
                                               Codes<float> cd) {
    const float keep = 1.0f - omega;
    for (int k = 0; k < kSpan<float>; k++) {
        const bool fuse = cd.at(k) == kTailInner ? inner : near;
        e.v[k] = fuse ? __fmaf_rn(omega, g.v[k], __fmul_rn(keep, e.v[k])) : __fmaf_rn(keep, e.v[k], __fmul_rn(omega, g.v[k]));
    }
    return e;
}
__device__ __forceinline__ Span<float> relaxed(const TailLevel<float>& L, float omega, Span<float> e, Span<float> g,
                                               const Codes<float>& cd) {
    return relaxed_as(L.fuse_inner, L.fuse_near, omega, e, g, cd);
}

// The sums of the unknown neighbours of a span's cells, in the order x left,
// right, y-1, y+1, z-1, z+1 (FP64: the three pairs first, which takes two of
// the seven 64-cycle operations off the chain).
template <class T>
__device__ __forceinline__ Span<T> neighbour_sums(const T* e, const Around<T>& at, const Codes<T>& cd) {
    constexpr int W = kSpan<T>;
    const Span<T> X = ldspan(e + at.i), A = ldspan(e + at.a), B = ldspan(e + at.b), D = ldspan(at.d), F = ldspan(at.f);
    const T h = e[at.h];
    Span<T> l, r, o;
#pragma unroll
    for (int k = 0; k < W; k++) {
        l.v[k] = at.O ? X.v[k] : (k == 0 ? h : X.v[k == 0 ? 0 : k - 1]);
        r.v[k] = at.O ? (k == W - 1 || k == at.last ? h : X.v[k == W - 1 ? k : k + 1]) : X.v[k];
    }
    if constexpr (W == 1) {
        const unsigned c = cd.w[0];
        const T x0 = (c & 3u) ? (T)0 : l.v[0], x1 = (c & 0xCu) ? (T)0 : r.v[0];
        const T y0 = (c & 0x30u) ? (T)0 : A.v[0], y1 = (c & 0xC0u) ? (T)0 : B.v[0];
        const T z0 = (c & 0x300u) ? (T)0 : D.v[0], z1 = (c & 0xC00u) ? (T)0 : F.v[0];
        o.v[0] = ((x0 + x1) + (y0 + y1)) + (z0 + z1);
    } else if (__all_sync(__activemask(), cd.inner())) {
#pragma unroll
        for (int k = 0; k < W; k++) o.v[k] = ((((l.v[k] + r.v[k]) + A.v[k]) + B.v[k]) + D.v[k]) + F.v[k];
    } else {
#pragma unroll
        for (int k = 0; k < W; k++) {
            const unsigned c = cd.at(k);
            T s = (c & 3u) ? (T)0 : l.v[k];
            s += (c & 0xCu) ? (T)0 : r.v[k];
            s += (c & 0x30u) ? (T)0 : A.v[k];
            s += (c & 0xC0u) ? (T)0 : B.v[k];
            s += (c & 0x300u) ? (T)0 : D.v[k];
            s += (c & 0xC00u) ? (T)0 : F.v[k];
            o.v[k] = s;
        }
    }
    return o;
}

// `sweeps` red-black sweeps of a level (B.inv[15] = 0 keeps e = 0 at cells that
// are not unknown).  Where every thread has at most one span of a colour, what
// the sweeps do not change -- the addresses, codes, diagonals, their inverses
// and h^2 r -- stays in registers (FP32 32^3: a half sweep 0.62 us; with the
// quotient's operands looked up in each of them 0.71, products alone 0.60).
template <class T>
__device__ __forceinline__ void tail_smooth(const TailLevel<T>& L, const Slab<T>& s, const Tables<T>& B,
                                            int sweeps, T omega, bool solo, cg::cluster_group& cl) {
    constexpr int W = kSpan<T>;
    const TailShape& S = L.s;
    const bool gs = omega == (T)1;
    const T h2 = L.h2;
    const int how = L.how, odd = L.odd;
    if (sweeps == 0) return;
    // (FP32: not with over-relaxation)
    bool resident = S.ny * S.zs <= S.rpi;
    if (resident) {
        const bool on = s.row0 < s.nrows;
        const int row = on ? s.row0 : 0, y = on ? s.y0 : 0, lz = on ? s.lz0 : 0;
        const Around<T> at0(S, s, 0, row, y, lz), at1(S, s, 1, row, y, lz);
        const int own = row * S.nxp + s.j0;
        const Codes<T> cd0(s.code + own), cd1(s.code + S.ploc + own);
        Span<T> r0 = ldspan(s.r + own), r1 = ldspan(s.r + S.ploc + own);
        Span<T> i0 = inverses<T>(B, cd0), i1 = inverses<T>(B, cd1);
        Span<T> d0, d1, c0, c1;  // (FP32: diagonals, and inverses where the quotient is taken)
        bool other = false;
#pragma unroll
        for (int k = 0; k < W; k++) {
            r0.v[k] *= h2;  // (exact: a power of two)
            r1.v[k] *= h2;
            if constexpr (W == 1) {  // (FP64: an operation less in each half sweep's chain)
                r0.v[k] *= i0.v[k];
                r1.v[k] *= i1.v[k];
            } else {
                d0.v[k] = B.diag[cd0.at(k) >> 12];
                d1.v[k] = B.diag[cd1.at(k) >> 12];
                c0.v[k] = how == kByTable ? (T)0 : B.cor[cd0.at(k) >> 12];
                c1.v[k] = how == kByTable ? (T)0 : B.cor[cd1.at(k) >> 12];
                other |= (cd0.at(k) >> 12) == kTailOdd || (cd1.at(k) >> 12) == kTailOdd;
            }
        }
        if constexpr (W == 4) {
            resident = gs;
            if (odd && __syncthreads_or(other)) {  // (rare)
                d0 = odd_diagonals(L.diag0, d0, cd0);
                d1 = odd_diagonals(L.diag0, d1, cd1);
                i0 = odd_inverses(d0, i0, cd0);
                i1 = odd_inverses(d1, i1, cd1);
                c0 = odd_inverses(d0, c0, cd0);
                c1 = odd_inverses(d1, c1, cd1);
            }
        }
        auto half = [&](const Around<T>& at, const Codes<T>& cd, const Span<T>& r, const Span<T>& id,
                        const Span<T>& dg, const Span<T>& cor, T* e) {
            if (on) {
                const Span<T> o = neighbour_sums<T>(s.e, at, cd);
                Span<T> g;
                if constexpr (W == 1) {
                    g.v[0] = o.v[0] * id.v[0] + r.v[0];
                    if (!gs) g = relaxed(L, omega, ldspan(e), g, cd);
                } else {
                    // (as quotients, all in registers and without a branch)
#pragma unroll
                    for (int k = 0; k < W; k++) {
                        const T n = r.v[k] + o.v[k];
                        g.v[k] = n * id.v[k];
                        g.v[k] = __fmaf_rn(__fmaf_rn(-g.v[k], dg.v[k], n), cor.v[k], g.v[k]);
                    }
                }
                stspan(e, g);
            }
            if (solo)
                __syncthreads();
            else
                cl.sync();
        };
        if (resident) {
            for (int h = 0; h < sweeps; h++) {
                half(at0, cd0, r0, i0, d0, c0, s.e + own);
                half(at1, cd1, r1, i1, d1, c1, s.e + S.ploc + own);
            }
            return;
        }
    }
    for (int h = 0; h < 2 * sweeps; h++) {
        const int colour = h & 1;
        s.rows(S, [&](int row, int y, int lz) {
            const int own = colour * S.ploc + row * S.nxp + s.j0;
            const Codes<T> cd(s.code + own);
            const Span<T> r = ldspan(s.r + own);
            const Span<T> o = neighbour_sums<T>(s.e, Around<T>(S, s, colour, row, y, lz), cd);
            Span<T> g;
#pragma unroll
            for (int k = 0; k < W; k++) g.v[k] = h2 * r.v[k] + o.v[k];
            g = quotients<T>(L, how, odd, B, g, inverses<T>(B, cd), cd);
            if (!gs) g = relaxed(L, omega, ldspan(s.e + own), g, cd);
            stspan(s.e + own, g);
        });
        if (solo)
            __syncthreads();
        else
            cl.sync();
    }
}

// One thread's bulk copies, completing on an mbarrier (bytes a multiple of
// 16, both addresses 16-byte aligned); the wait is bounded (about a second).
__device__ __forceinline__ void bulk_expect(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_in(void* dst, const void* src, unsigned bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool bulk_wait(unsigned bar, unsigned parity) {
    const long long t0 = clock64();
    for (;;) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > (1LL << 31)) return false;
    }
}

// Natural cell of place j (x parity O) of row (y, z), and where level l0's
// global arrays hold it.
__device__ __forceinline__ int global_place(const TailShape& S, int half, int colour, int x, int y, int z) {
    const int c = x + S.nx * (y + S.ny * z);
    return half ? colour * half + (c >> 1) : c;
}

template <class T>
__global__ void __launch_bounds__(kTailThreads) k_tail(const __grid_constant__ TailArgs<T> A) {
    constexpr int W = kSpan<T>;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ T inv_tab[ES_MAXLEV][16], diag_tab[ES_MAXLEV][16], cor_tab[sizeof(T) == 4 ? ES_MAXLEV : 1][16];
    __shared__ __align__(8) uint64_t bar;
    __shared__ int late;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    // The stencil codes (the mapping's, at least two kernels back), the zero
    // iterates and the diagonals, before the wait for the kernel before this one.
    const unsigned bar_at = (unsigned)__cvta_generic_to_shared(&bar);
    if (threadIdx.x == 0) {
        late = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_at) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        bulk_expect(bar_at, A.code_bytes);
        bulk_in(smem, A.codes + (size_t)rank * A.code_bytes, A.code_bytes, bar_at);
    }
    for (int t = threadIdx.x; t < 16 * A.n; t += kTailThreads) {
        const int l = t >> 4, k = t & 15;
        const T d = A.lv[l].diag0 + (T)(k == (int)kTailEven ? 0 : k - 6), y = k == 15 ? (T)0 : (T)1 / d;
        diag_tab[l][k] = d;
        inv_tab[l][k] = y;
        if constexpr (sizeof(T) == 4) cor_tab[l][k] = k == 6 && A.lv[l].how == kNearQuotient ? (T)0 : y;
    }
    for (int t = A.code_bytes + 16 * (int)threadIdx.x; t < A.smem_bytes; t += 16 * kTailThreads)
        *reinterpret_cast<uint4*>(smem + t) = make_uint4(0u, 0u, 0u, 0u);
    // (these stores go through the generic proxy; the bulk copies below, which
    // overwrite some of them, through the async one)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && !bulk_wait(bar_at, 0)) late = 1;
    pdl_wait();
    auto tables = [&](int l) { return Tables<T>{inv_tab[l], diag_tab[l], cor_tab[sizeof(T) == 4 ? l : 0]}; };
    {
        const TailShape& S = A.lv[0].s;
        const Slab<T> s(S, smem, cl, rank);
        if (A.half && S.nxp == S.nxh && !A.warm) {
            // a colour's slab is one run of the colour-split right-hand side
            if (threadIdx.x == 0 && s.nzl > 0) {
                const unsigned bytes = (unsigned)(s.nzl * S.plane * sizeof(T));
                const T* src = A.rhs + (size_t)s.z0 * S.plane;
                bulk_expect(bar_at, 2 * bytes);
                bulk_in(s.r, src, bytes, bar_at);
                bulk_in(s.r + S.ploc, src + A.half, bytes, bar_at);
                if (!bulk_wait(bar_at, 1)) late = 1;
            }
            __syncthreads();
        } else {
            __syncthreads();
            // both colours' spans of a row at once: natural cells 2 j0 .. 2 j0 + 2 W - 1
            s.rows(S, [&](int row, int y, int lz) {
                const int O = (y + s.z0 + lz) & 1, own = row * S.nxp + s.j0;
                const Codes<T> cd[2] = {Codes<T>(s.code + own), Codes<T>(s.code + S.ploc + own)};
                Span<T> r[2], e[2];
#pragma unroll
                for (int k = 0; k < W; k++)
#pragma unroll
                    for (int q = 0; q < 2; q++) {
                        const bool on = cd[q].at(k) != kTailOff;
                        const int g = global_place(S, A.half, q, 2 * (s.j0 + k) + (q ? 1 - O : O), y, s.z0 + lz);
                        r[q].v[k] = on ? A.rhs[g] : (T)0;
                        e[q].v[k] = on && A.warm ? A.out[g] : (T)0;
                    }
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    stspan(s.r + q * S.ploc + own, r[q]);
                    if (A.warm) stspan(s.e + q * S.ploc + own, e[q]);
                }
            });
        }
    }
    if (late && threadIdx.x == 0) atomicOr(A.status, DS_TIMEOUT);
    cl.sync();
    for (int l = 0; l + 1 < A.n; l++) {
        const TailLevel<T>& L = A.lv[l];
        const TailShape& S = L.s;
        const TailShape& M = A.lv[l + 1].s;
        const Slab<T> s(S, smem, cl, rank);
        tail_smooth<T>(L, s, tables(l), A.nu1, A.omega, false, cl);
        // restriction: the mean of the 8 children's residuals (with red_only
        // the black ones count as 0); the children of a coarse cell share a slab
        // (an even number of planes), the coarse cell may be another block's.
        // A thread owns the coarse cells of a row above a span of each fine row.
        const int cny = S.ny >> 1;
        T* cr = (T*)(smem + M.r);
        const int ncr = cny * (s.nzl >> 1);
        if (s.row0 < S.rpi)
            for (int crow = s.row0; crow < ncr; crow += S.rpi) {
                const int Zl = (int)(((unsigned)crow * M.mny) >> 22), Y = crow - Zl * cny;  // (cny = M.ny)
                T sum[W];
#pragma unroll
                for (int k = 0; k < W; k++) sum[k] = (T)0;
#pragma unroll 2
                for (int q = 0; q < 4; q++) {
                    const int y = 2 * Y + (q & 1), lz = 2 * Zl + (q >> 1), row = y + S.ny * lz;
                    T res[2][W];  // the even-x and the odd-x children
#pragma unroll
                    for (int d = 0; d < 2; d++) {
                        const int colour = (d + y + s.z0 + lz) & 1;
                        const int own = colour * S.ploc + row * S.nxp + s.j0;
#pragma unroll
                        for (int k = 0; k < W; k++) res[d][k] = (T)0;
                        if (L.red_only && colour) continue;
                        const Codes<T> cd(s.code + own);
                        const Span<T> o = neighbour_sums<T>(s.e, Around<T>(S, s, colour, row, y, lz), cd);
                        const Span<T> r = ldspan(s.r + own), e = ldspan(s.e + own);
#pragma unroll
                        for (int k = 0; k < W; k++) {
                            const unsigned c = cd.at(k);
                            T dg = diag_tab[l][c >> 12];
                            if constexpr (W == 4)
                                if ((c >> 12) == kTailOdd) dg = code_diag(L.diag0, c);
                            if (c != kTailOff) res[d][k] = r.v[k] - (dg * e.v[k] - o.v[k]) * L.inv_h2;
                        }
                    }
#pragma unroll
                    for (int k = 0; k < W; k++)
                        sum[k] = L.pairs ? sum[k] + (res[0][k] + res[1][k]) : (sum[k] + res[0][k]) + res[1][k];
                }
                const int Z = (s.z0 >> 1) + Zl, owner = slab_owner(M, Z);
                T* out = cl.map_shared_rank(cr, owner) + M.nxp * (Y + M.ny * (Z - owner * M.zs));
#pragma unroll
                for (int k = 0; k < W; k++) {
                    const int X = s.j0 + k;
                    if ((X >> 1) < M.nxp) out[((X + Y + Z) & 1) * M.ploc + (X >> 1)] = sum[k] * (T)0.125;
                }
            }
        cl.sync();
    }
    {
        const TailLevel<T>& L = A.lv[A.n - 1];
        if (!A.solo || rank == 0)
            tail_smooth<T>(L, Slab<T>(L.s, smem, cl, rank), tables(A.n - 1), A.sweeps, A.omega, A.solo != 0, cl);
        if (A.solo) cl.sync();
    }
    for (int l = A.n - 2; l >= 0; l--) {
        const TailLevel<T>& L = A.lv[l];
        const TailShape& S = L.s;
        const TailShape& M = A.lv[l + 1].s;
        const Slab<T> s(S, smem, cl, rank);
        // piecewise-constant prolongation into unknown cells (e is 0 at parents
        // that are not unknown); ahead of a Gauss-Seidel sweep the black cells
        // only: it replaces the red ones without reading them
        const T* ce = (const T*)(smem + M.e);
        for (int colour = A.omega == (T)1 && A.nu2 >= 1 ? 1 : 0; colour < 2; colour++)
            s.rows(S, [&](int row, int y, int lz) {
                const int i = colour * S.ploc + row * S.nxp + s.j0;
                const int Y = y >> 1, Z = (s.z0 + lz) >> 1, owner = slab_owner(M, Z);
                const T* p = cl.map_shared_rank(ce, owner) + M.nxp * (Y + M.ny * (Z - owner * M.zs));
                const Codes<T> cd(s.code + i);
                Span<T> v = ldspan(s.e + i);
#pragma unroll
                for (int k = 0; k < W; k++) {
                    const int X = s.j0 + k;
                    if (cd.at(k) != kTailOff) v.v[k] += p[((X + Y + Z) & 1) * M.ploc + (X >> 1)];
                }
                stspan(s.e + i, v);
            });
        cl.sync();
        tail_smooth<T>(L, s, tables(l), A.nu2, A.omega, false, cl);
    }
    {
        const TailShape& S = A.lv[0].s;
        const Slab<T> s(S, smem, cl, rank);
        if (A.half && S.nxp == S.nxh) {
            // (0 at cells that are not unknown: nobody reads them)
            if (threadIdx.x == 0 && s.nzl > 0) {
                const unsigned bytes = (unsigned)(s.nzl * S.plane * sizeof(T));
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                for (int colour = 0; colour < 2; colour++)
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                                     A.out + (size_t)colour * A.half + (size_t)s.z0 * S.plane),
                                 "r"((unsigned)__cvta_generic_to_shared(s.e + colour * S.ploc)), "r"(bytes)
                                 : "memory");
                asm volatile("cp.async.bulk.commit_group;\ncp.async.bulk.wait_group 0;" ::: "memory");
            }
        } else {
            s.rows(S, [&](int row, int y, int lz) {
                const int O = (y + s.z0 + lz) & 1, own = row * S.nxp + s.j0;
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const Codes<T> cd(s.code + q * S.ploc + own);
                    const Span<T> e = ldspan(s.e + q * S.ploc + own);
#pragma unroll
                    for (int k = 0; k < W; k++)
                        if (cd.at(k) != kTailOff)
                            A.out[global_place(S, A.half, q, 2 * (s.j0 + k) + (q ? 1 - O : O), y, s.z0 + lz)] = e.v[k];
                }
            });
        }
    }
    // (every block's reads of another's shared memory ended before its last
    // barrier, except after no sweep at all)
    cl.sync();
}

// The codes of all levels in the blocks' layout: a thread a span of four
// places (blockIdx.y: level).
__global__ void __launch_bounds__(256) k_tail_codes(const __grid_constant__ TailCodes A) {
    pdl_wait();
    const TailShape& S = A.s[blockIdx.y];
    const uint8_t* st = A.st[blockIdx.y];
    const int spans = S.ploc / 4;  // of a colour in a slab
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < 2 * spans * A.blocks; t += gridDim.x * blockDim.x) {
        const int block = t / (2 * spans), q = t - 2 * spans * block;
        const int colour = q >= spans ? 1 : 0, i = q - colour * spans;
        const int pw = S.nxp / 4, row = i / pw, j0 = 4 * (i - row * pw);
        const int lz = row / S.ny, y = row - lz * S.ny, z = block * S.zs + lz;
        const int O = (colour + y + z) & 1;
        unsigned code[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int x = 2 * (j0 + k) + O;
            code[k] = kTailOff;
            if (z >= S.nz || j0 + k >= S.nxh || x >= S.nx) continue;
            const int c = x + S.nx * (y + S.ny * z);
            if ((st[c] & ST_KIND) != ST_UNKNOWN) continue;
            const int v[3] = {x, y, z}, n3[3] = {S.nx, S.ny, S.nz}, stride[3] = {1, S.nx, S.nx * S.ny};
            unsigned kind[6], wall = 0;
#pragma unroll
            for (int f = 0; f < 6; f++) {
                const int a = f >> 1;
                int p = v[a] + ((f & 1) ? 1 : -1);
                if (p < 0 || p >= n3[a]) {
                    if (!A.per[a]) wall |= 1u << f;
                    p = p < 0 ? p + n3[a] : p - n3[a];
                }
                kind[f] = st[c + (p - v[a]) * stride[a]];
            }
            unsigned cd = 0;
            int dk = 6;
#pragma unroll
            for (int f = 0; f < 6; f++) {
                const unsigned u =
                    ((wall >> f) & 1u) ? (A.pot_bc[f] == ES_POT_DIRICHLET ? 1u : 2u) : (kind[f] & ST_KIND);
                cd |= u << (2 * f);
                dk += u == 0u ? 0 : (u == 1u ? 1 : -1);
            }
            if (A.diag0[blockIdx.y] > 0.0f && cd != 0u)
                dk = code_diag(A.diag0[blockIdx.y], cd) != A.diag0[blockIdx.y] + (float)(dk - 6)
                         ? (int)kTailOdd
                         : (dk == 6 ? (int)kTailEven : dk);
            code[k] = cd | ((unsigned)dk << 12);
        }
        *reinterpret_cast<uint2*>(A.out + (size_t)block * A.bytes + S.c + 2 * (size_t)(colour * S.ploc + 4 * i)) =
            make_uint2(code[0] | (code[1] << 16), code[2] | (code[3] << 16));
    }
}

// The levels l0 .. L-1 in a cluster of `blocks`: their shapes and places in a
// block's shared memory (codes first, then e and the right-hand sides).
struct TailPlan {
    TailShape s[ES_MAXLEV];
    int n, blocks, solo, code_bytes, smem_bytes;
};

bool tail_layout(const es_params& P, int l0, TailPlan& T) {
    const int ts = P.precision == ES_FP64 ? 8 : 4;
    T.n = P.levels - l0;
    T.blocks = kTailCluster;
    const int* d = P.dims;
    const int cl = P.levels - 1;
    const long long N = (long long)(d[0] >> l0) * (d[1] >> l0) * (d[2] >> l0);
    const long long Nc = (long long)(d[0] >> cl) * (d[1] >> cl) * (d[2] >> cl);
    if (N > (ts == 8 ? kTailCells64 : kTailCells32)) return false;
    T.solo = Nc <= (ts == 8 ? 64 : 4096) ? 1 : 0;
    long long at = 0;
    for (int l = 0; l < T.n; l++) {
        TailShape& S = T.s[l];
        S.nx = d[0] >> (l0 + l);
        S.ny = d[1] >> (l0 + l);
        S.nz = d[2] >> (l0 + l);
        S.nxh = (S.nx + 1) / 2;
        S.nxp = (S.nxh + 3) / 4 * 4;
        S.pw = S.nxp / (ts == 8 ? kSpan<double> : kSpan<float>);
        if (S.pw > kTailThreads || S.ny > 1024 || S.nz > 1023) return false;
        // an even number of planes, so that the children of a coarse plane share
        // a block (the coarsest level has none)
        S.zs = l + 1 < T.n ? 2 * ((S.nz / 2 + T.blocks - 1) / T.blocks)
                           : (T.solo ? S.nz : (S.nz + T.blocks - 1) / T.blocks);
        const long long block = (long long)S.nx * S.ny * S.zs;  // cells of a slab
        const bool last = l + 1 == T.n;
        // (a coarsest level that one block would hold otherwise, k_coarse_solve,
        // is here in any case)
        if (!(last && Nc * (2 * ts + 1) <= kCoarseSmem) &&
            block > (ts == 8 ? (last ? kTailLast64 : kTailBlock64) : (last ? kTailLast32 : kTailBlock32)))
            return false;
        S.plane = S.nxp * S.ny;
        if ((long long)S.zs * S.plane * (2 * ts + 2) * 2 > (long long)kTailSmem) return false;
        S.ploc = S.zs * S.plane;
        S.rpi = kTailThreads / S.pw;
        S.dz = S.rpi / S.ny;
        S.dy = S.rpi - S.dz * S.ny;
        S.mpw = ((1u << 22) + S.pw - 1) / S.pw;
        S.mny = ((1u << 22) + S.ny - 1) / S.ny;
        S.mzs = ((1u << 22) + S.zs - 1) / S.zs;
        S.c = (int)at;
        at += (4LL * S.ploc + 15) & ~15LL;
    }
    T.code_bytes = (int)at;
    for (int l = 0; l < T.n; l++) {
        TailShape& S = T.s[l];
        S.e = (int)at;
        S.r = (int)(at + 2LL * S.ploc * ts);
        at += 4LL * S.ploc * ts;
        if (at > (long long)kTailSmem) return false;
    }
    T.smem_bytes = (int)at;
    return true;
}

// The finest level whose coarser ones all fit the cluster, or -1.  A cell of a
// periodic axis of one cell is its own neighbour there, of its own colour,
// which the colours' separate arrays do not hold in the neighbour's place:
// such grids (one level) are launched.
int tail_first(const es_params& P, TailPlan& T) {
    if (P.phi_t > 0.0 || P.smoother != ES_SMOOTH_TWO_PASS) return -1;
    for (int a = 0; a < 3; a++)
        if (P.periodic[a] && P.dims[a] == 1) return -1;
    const long long most = P.near_list_cells > 0 ? (long long)P.near_list_cells : (long long)ES_NEAR_LIST_CELLS;
    for (int l = P.mg_storage == ES_MG_FP16 ? 1 : 0; l < P.levels; l++) {
        if ((long long)(P.dims[0] >> l) * (P.dims[1] >> l) * (P.dims[2] >> l) > most) continue;
        if (tail_layout(P, l, T)) return l;
    }
    return -1;
}

}  // namespace

bool tail_split(const es_ctx* c) {
    const int l0 = c->tail_l0;
    return l0 >= 1 && l0 < c->L && split_level(c, l0 - 1) && c->ln[l0][0] % 8 == 0;
}

namespace {

template <class T>
cudaError_t tail_run(es_ctx* c, int warm) {
    TailPlan p;
    const int l0 = c->tail_l0;
    tail_layout(c->P, l0, p);
    TailArgs<T> A;
    A.n = p.n;
    for (int l = 0; l < p.n; l++) {
        const double h = (double)(1 << (l0 + l));
        TailLevel<T>& L = A.lv[l];
        L = TailLevel<T>{p.s[l], (T)(h * h), (T)(1.0 / (h * h)), (T)(6.0 + c->S.kappa * c->S.kappa * h * h)};
        L.how = kByTable;
        L.odd = 0;
        L.red_only = c->P.omega == 1.0 && c->P.nu1 >= 1;
        L.pairs = 1;
        L.fuse_inner = L.fuse_near = 0;
        if (sizeof(T) == 4) {
            // what the level's kernels do when it is launched by itself
            const bool spans = p.s[l].nx % 4 == 0;
            for (int k = -6; k <= 6; k++) L.odd |= (double)(T)((double)L.diag0 + k) != (double)L.diag0 + k;
            L.how = spans ? kNearQuotient : kQuotient;
            if (l + 1 < p.n || coarse_divides(c) == 2) {
                L.fuse_inner = !spans;                         // (k_smooth)
                L.fuse_near = !spans || split_level(c, l0 + l);  // (near_gs)
            } else {
                L.how = coarse_divides(c) == 0 ? kByTable : kQuotient;
                if (L.how == kByTable) L.odd = 0;
            }
            L.red_only = L.red_only && spans;
            L.pairs = spans;
        }
    }
    A.codes = c->tail_codes;
    A.code_bytes = p.code_bytes;
    A.smem_bytes = p.smem_bytes;
    A.rhs = (const T*)c->rhs[l0];
    A.out = (T*)c->e[l0];
    A.half = split_level(c, l0) || tail_split(c) ? c->ln[l0][0] * c->ln[l0][1] * c->ln[l0][2] / 2 : 0;
    A.warm = warm && A.n > 1;  // (a single level starts from zero)
    A.nu1 = c->P.nu1;
    A.nu2 = c->P.nu2;
    A.sweeps = c->P.coarse_sweeps;
    A.omega = (T)c->P.omega;
    A.solo = p.solo;
    A.status = c->d_status;
    double cells = 0.0;
    for (int l = l0; l < c->L; l++) cells += (double)c->ln[l][0] * c->ln[l][1] * c->ln[l][2];
    ProfScope ps(c, "tail", l0, cells * (2.0 * sizeof(T) + 1.0));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.blocks);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = p.smem_bytes;
    cfg.stream = c->stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = p.blocks;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_tail<T>, A);
    count(c);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

size_t tail_code_bytes(const es_params* P) {
    TailPlan T;
    return tail_first(*P, T) < 0 ? 0 : (size_t)T.blocks * T.code_bytes;
}

// Once a context: the levels that k_tail takes, the kernel's shared memory
// and cluster size (both belong to the kernel and are set to the most any
// context needs), and whether the device can place such a cluster at all;
// without it the levels are launched one by one.
void tail_setup(es_ctx* c) {
    TailPlan T;
    c->tail_l0 = c->L;
    const int l0 = tail_first(c->P, T);
    if (l0 < 0) return;
    const void* k = mixed(c) ? (const void*)k_tail<float> : (const void*)k_tail<double>;
    bool ok = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmem) == cudaSuccess &&
              cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    if (ok) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(T.blocks);
        cfg.blockDim = dim3(kTailThreads);
        cfg.dynamicSmemBytes = kTailSmem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = T.blocks;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        ok = cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0;
    }
    if (ok)
        c->tail_l0 = l0;
    else
        cudaGetLastError();
}

cudaError_t launch_tail(es_ctx* c, int warm) { return mixed(c) ? tail_run<float>(c, warm) : tail_run<double>(c, warm); }

// After the coarse states of a mapping.
cudaError_t launch_tail_codes(es_ctx* c) {
    if (c->tail_l0 >= c->L) return cudaSuccess;
    TailPlan p;
    tail_layout(c->P, c->tail_l0, p);
    TailCodes A;
    A.n = p.n;
    A.blocks = p.blocks;
    A.bytes = p.code_bytes;
    for (int l = 0; l < p.n; l++) {
        A.s[l] = p.s[l];
        A.st[l] = c->st[c->tail_l0 + l];
        const double h = (double)(1 << (c->tail_l0 + l));
        const bool table = l + 1 == p.n && coarse_divides(c) == 0;  // (k_coarse_lists takes the sum's inverse)
        A.diag0[l] = mixed(c) && !table ? (float)(6.0 + c->S.kappa * c->S.kappa * h * h) : 0.0f;
    }
    for (int a = 0; a < 3; a++) A.per[a] = c->g.per[a];
    for (int f = 0; f < 6; f++) A.pot_bc[f] = c->S.pot_bc[f];
    A.out = c->tail_codes;
    const int spans = p.s[0].ploc / 2 * p.blocks;
    launch_pdl(c, k_tail_codes, dim3((spans + 255) / 256, p.n), 256, 0, A);
    count(c);
    return cudaGetLastError();
}

}  // namespace es
