// es_lbm.cu -- fused stream-collide (a7), momentum-exchange force/torque (a8)
// and rigid-body update (a9); Sec. 4.1, Sec. 4.2, Sec. 5.7.
//
// Stream-collide is a single pull sweep over a structure-of-arrays PDF
// field: a thread per cell gathers f_q(x) = f~_q(x - e_q) from the 19
// streams (a warp reads 32 consecutive cells of each stream; the +-x
// shifted streams are one element off and are served by the same L1/L2
// sectors), collides in registers and writes its 19 populations.  Cells
// next to an obstacle or a wall (F_NEAR19) take the moving bounce-back of
// Eq. LBMMovWall instead of the pull for the affected directions.
//
// MIXED32 stores f_q - w_q in float: the collision is linear in f, and the
// weights cancel in every term except the density, which becomes 1 + sum.
#include <cmath>
#include <type_traits>

#include "es_device.cuh"

namespace es {

namespace {

// Base pointers of the 19 source and destination streams, so that an access
// is a 32-bit cell offset from a base (no 64-bit products in the kernel).
template <class S>
struct Streams {
    const S* src[19];
    S* dst[19];
};

// Float copy of the particle state used by the FP32 stream-collide (centre,
// velocity, angular velocity), so that its moving-wall term needs no FP64:
// made at creation, then kept by the kernels that change the state.
__global__ void k_particles_f32(int np, const DParticle* __restrict__ part, float* __restrict__ pf) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    for (int a = 0; a < 3; a++) {
        pf[12 * p + a] = (float)part[p].x[a];
        pf[12 * p + 3 + a] = (float)part[p].v[a];
        pf[12 * p + 6 + a] = (float)part[p].w[a];
    }
}

// A population whose pull source lies beyond a non-periodic face (walls
// half-way outside the first and last layer): the direction and cell it is
// taken from.  No-slip face: resting bounce-back, the cell's own population
// of the opposite direction.  Free-slip (every crossed face free-slip):
// specular reflection; the population arriving with e_q left the fluid cell
// s = x - (the components of e_q parallel to the crossed faces) in the
// direction with the crossed components reversed.  An obstacle cell at s
// falls back to bounce-back.  Either direction has the weight of q.
struct WallSrc {
    int q;
    long long cell;
};

__device__ __forceinline__ WallSrc wall_source(const Grid& g, int slip_faces, const int32_t* __restrict__ owner,
                                               int x, int y, int z, int q, long long c) {
    const int cv[3] = {cx(q), cy(q), cz(q)};
    const int p[3] = {x, y, z};
    const int n[3] = {g.nx, g.ny, g.nz};
    int m[3], s[3];
    bool slip = true;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int v = p[a] - cv[a];
        if (cv[a] != 0 && !g.per[a] && (v < 0 || v >= n[a])) {
            slip = slip && ((slip_faces >> (2 * a + (v >= n[a] ? 1 : 0))) & 1);
            m[a] = -cv[a];
            s[a] = p[a];
        } else {
            m[a] = cv[a];
            s[a] = v < 0 ? v + n[a] : (v >= n[a] ? v - n[a] : v);
        }
    }
    if (slip) {
        const long long sc = lin(g, s[0], s[1], s[2]);
        if (owner[sc] < 0) {
            int qm = 0;
#pragma unroll
            for (int k = 1; k < 19; k++)
                if (cx(k) == m[0] && cy(k) == m[1] && cz(k) == m[2]) qm = k;
            return WallSrc{qm, sc};
        }
    }
    return WallSrc{opp(q), c};
}

// The collision's constants, formed once on the host from the TRT rates
// (Sec. 4.1) and the factors 1 + lambda / 2 that go with the modified velocity.
template <class C>
struct Trt {
    C rest;        // 1 + lambda_e
    C se, so;      // (1 + lambda_e) / 2, (1 + lambda_o) / 2
    C kr, ku, kf;  // -lambda_e, 1.5 lambda_e, -3 (1 + lambda_e / 2)
    C hu, hf;      // w_1 (-4.5 lambda_e), w_1 9 (1 + lambda_e / 2)
    C gu, gf;      // w_1 (-3 lambda_o), w_1 3 (1 + lambda_o / 2)
    C lam_e, lam_o;  // the rates themselves (collide_direct)
};

template <class C>
Trt<C> trt(double le, double lo) {
    const double ae = 1.0 + 0.5 * le, ao = 1.0 + 0.5 * lo, w1 = wq(1);
    return Trt<C>{(C)(1.0 + le),       (C)(0.5 + 0.5 * le), (C)(0.5 + 0.5 * lo),  (C)(-le),
                  (C)(1.5 * le),       (C)(-3.0 * ae),      (C)(-4.5 * le * w1),  (C)(9.0 * ae * w1),
                  (C)(-3.0 * lo * w1), (C)(3.0 * ao * w1),  (C)le,               (C)lo};
}

// TRT collision of one cell from its pulled populations f (working values)
// and its body force plus acceleration: the moments (Eq. MacroscopVel) with
// the modified velocity (Eq. modified_velocity), the even and odd parts of
// Eq. TRTOp with the incompressible equilibrium (Eq. EqPDF_TRT) and Luo's
// forcing (Eq. LBE_forcetermLuo), split into even w(9 cu cf - 3 u.f) and odd
// 3 w cf; put(q, v) receives each post-collision value.  Every
// stream-collide kernel of a form calls the same function, so all give the
// same bits.
//
// The FP64 kernel is bound by the FP64 pipe (2 operations a clock and SM),
// so the number of operations is what counts.  With the sums p = f_q + f_-q
// and differences m = f_q - f_-q of the nine pairs, the moments need 39
// additions instead of 48, and a pair becomes s +- d with
//   s = (1 + lambda_e)/2 p + w (K + (c.u)(c.h)),  h = -4.5 lambda_e u + 9 ae F,
//   K = -lambda_e rho + 1.5 lambda_e u.u - 3 ae u.F,
//   d = (1 + lambda_o)/2 m + w c.g,               g = -3 lambda_o u + 3 ao F
// (ae, ao = 1 + lambda / 2; w_2 = w_1 / 2 folded into h, K and g): 139
// operations a cell instead of 357 (a 160 x 136 x 152 FP64 step: 1.88 ms
// before, 0.96 ms with it, 0.90 ms with the one surface velocity a cell of
// lbm_cell).
template <class C, class Put>
__device__ __forceinline__ void collide(const C (&f)[19], C fx, C fy, C fz, const Trt<C>& R, Put&& put) {
    C p[10], m[10];
#pragma unroll
    for (int q = 1; q <= 9; q++) {
        p[q] = f[q] + f[q + 9];
        m[q] = f[q] - f[q + 9];
    }
    // in the shifted form rho holds rho - 1; w_q * rho below is then the
    // shifted equilibrium directly
    C rho = f[0], jx = (C)0, jy = (C)0, jz = (C)0;
#pragma unroll
    for (int q = 1; q <= 9; q++) rho += p[q];
#pragma unroll
    for (int q = 9; q >= 1; q--) {  // (the small diagonal parts first)
        if (cx(q)) jx += cx(q) > 0 ? m[q] : -m[q];
        if (cy(q)) jy += cy(q) > 0 ? m[q] : -m[q];
        if (cz(q)) jz += cz(q) > 0 ? m[q] : -m[q];
    }
    const C u[3] = {jx + (C)0.5 * fx, jy + (C)0.5 * fy, jz + (C)0.5 * fz};
    const C F[3] = {fx, fy, fz};
    const C uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const C uf = u[0] * fx + u[1] * fy + u[2] * fz;
    const C K1 = (C)wq(1) * (R.kr * rho + R.ku * uu + R.kf * uf), K2 = (C)0.5 * K1;
    put(0, R.rest * f[0] + (C)6 * K1);  // (w_0 = 6 w_1)
    C h[3], g[3], h2[3], g2[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        h[a] = R.hu * u[a] + R.hf * F[a];
        g[a] = R.gu * u[a] + R.gf * F[a];
        h2[a] = (C)0.5 * h[a];
        g2[a] = (C)0.5 * g[a];
    }
#pragma unroll
    for (int q = 1; q <= 9; q++) {
        C ev, od;
        if (q <= 3) {
            ev = K1 + u[q - 1] * h[q - 1];
            od = g[q - 1];
        } else {
            // the direction's two axes, the first with coefficient +1
            const int a = cx(q) ? 0 : 1, b = cz(q) ? 2 : 1;
            const bool plus = (b == 1 ? cy(q) : cz(q)) > 0;
            ev = K2 + (plus ? u[a] + u[b] : u[a] - u[b]) * (plus ? h2[a] + h2[b] : h2[a] - h2[b]);
            od = plus ? g2[a] + g2[b] : g2[a] - g2[b];
        }
        const C s = R.se * p[q] + ev, d = R.so * m[q] + od;
        put(q, s + d);
        put(q + 9, s - d);
    }
}

// The same collision term by term, for the reduced forms, whose rounding is
// what decides their error: with these operations the FP16 form's 32^3
// sphere is 8.6e-5 from the FP64 oracle's velocity after 100 steps, with those
// of collide() 1.2e-4, and their FP32 kernels are bound by HBM (512^3 MIXED32:
// 3.89 ms against 3.85).
template <class C, class Put>
__device__ __forceinline__ void collide_direct(const C (&f)[19], C fx, C fy, C fz, C lam_e, C lam_o, Put&& put) {
    // moments (Eq. MacroscopVel) with the modified velocity (Eq. modified_velocity)
    C rho = (C)0, jx = (C)0, jy = (C)0, jz = (C)0;
#pragma unroll
    for (int q = 0; q < 19; q++) {
        rho += f[q];
        if (cx(q)) jx += cx(q) > 0 ? f[q] : -f[q];
        if (cy(q)) jy += cy(q) > 0 ? f[q] : -f[q];
        if (cz(q)) jz += cz(q) > 0 ? f[q] : -f[q];
    }
    // in the shifted form rho holds rho - 1; w_q * rho below is then the
    // shifted equilibrium directly
    const C ux = jx + (C)0.5 * fx, uy = jy + (C)0.5 * fy, uz = jz + (C)0.5 * fz;
    const C uu = ux * ux + uy * uy + uz * uz;
    const C uf = ux * fx + uy * fy + uz * fz;
    const C ae = (C)1 + (C)0.5 * lam_e, ao = (C)1 + (C)0.5 * lam_o;

    // rest population: even part only
    {
        const C w0 = (C)wq(0);
        const C eq0 = w0 * (rho - (C)1.5 * uu);
        const C F0 = w0 * ((C)-3 * uf);
        put(0, f[0] + lam_e * (f[0] - eq0) + ae * F0);
    }
    // pairs (q, q+9): TRT split into even and odd parts (Eq. TRTOp, Eq. EqPDF_TRT)
#pragma unroll
    for (int q = 1; q <= 9; q++) {
        const C w = (C)wq(q);
        const C cu = (C)cx(q) * ux + (C)cy(q) * uy + (C)cz(q) * uz;
        const C cf = (C)cx(q) * fx + (C)cy(q) * fy + (C)cz(q) * fz;
        const C eq_e = w * (rho + (C)4.5 * cu * cu - (C)1.5 * uu);
        const C eq_o = w * (C)3 * cu;
        const C fe = (C)0.5 * (f[q] + f[q + 9]);
        const C fo = (C)0.5 * (f[q] - f[q + 9]);
        // Luo's term (Eq. LBE_forcetermLuo) split: even w(9 cu cf - 3 u.f), odd 3 w cf,
        // with the (1 + lambda/2) factors that go with the modified velocity
        const C Fe = w * ((C)9 * cu * cf - (C)3 * uf);
        const C Fo = w * (C)3 * cf;
        const C even = lam_e * (fe - eq_e) + ae * Fe;
        const C odd = lam_o * (fo - eq_o) + ao * Fo;
        put(q, f[q] + even + odd);
        put(q + 9, f[q + 9] + even - odd);
    }
}

// c_q . u (no operations for the components that are 0).
__device__ __forceinline__ double dot_c(int q, const double (&u)[3]) {
    const int c[3] = {cx(q), cy(q), cz(q)};
    double t = 0.0;
    bool some = false;
#pragma unroll
    for (int a = 0; a < 3; a++)
        if (c[a]) {
            t = some ? (c[a] > 0 ? t + u[a] : t - u[a]) : (c[a] > 0 ? u[a] : -u[a]);
            some = true;
        }
    return t;
}

// The faces (bits as in lbm_cell) beyond which the source x - c_q lies of a
// cell at all of them.
__device__ __forceinline__ unsigned crossed(int q) {
    return (cx(q) > 0 ? 1u : cx(q) < 0 ? 2u : 0u) | (cy(q) > 0 ? 4u : cy(q) < 0 ? 8u : 0u) |
           (cz(q) > 0 ? 16u : cz(q) < 0 ? 32u : 0u);
}

// The electric body force evaluated inside the stream-collide (reduced
// forms): psi (the float potential), E_ext and kappa^2 eps.
struct FbPsi {
    const float* psi;
    float Ex, Ey, Ez, k2e;
};

// psi at an interior cell and its 18 neighbours; sx, sy, sz: the offsets of
// the steps +1, 0, -1 along each axis (wrapped), p the cell's own value.
__device__ __forceinline__ Psi19 load_psi19(const float* __restrict__ p, const int (&sx)[3], const int (&sy)[3],
                                            const int (&sz)[3]) {
    return Psi19{__ldg(p),
                 __ldg(p + sx[0]),
                 __ldg(p + sx[2]),
                 __ldg(p + sy[0]),
                 __ldg(p + sy[2]),
                 __ldg(p + sz[0]),
                 __ldg(p + sz[2]),
                 __ldg(p + sx[0] + sy[0]),
                 __ldg(p + sx[2] + sy[2]),
                 __ldg(p + sx[0] + sy[2]),
                 __ldg(p + sx[2] + sy[0]),
                 __ldg(p + sx[0] + sz[0]),
                 __ldg(p + sx[2] + sz[2]),
                 __ldg(p + sx[0] + sz[2]),
                 __ldg(p + sx[2] + sz[0]),
                 __ldg(p + sy[0] + sz[0]),
                 __ldg(p + sy[2] + sz[2]),
                 __ldg(p + sy[0] + sz[2]),
                 __ldg(p + sy[2] + sz[0])};
}

// SLIP: the grid has free-slip faces (a separate instance, so that the
// common no-slip/periodic form keeps its register count).  FBPSI: the body
// force of an interior fluid cell (no obstacle or wall among its D3Q19
// neighbours) is formed here from the potential at the cell and its 18
// neighbours (body_force_iso, Sec. 5.6), so f_b makes no round trip through
// HBM: the cell reads 4 bytes of psi (the neighbours' come from cache)
// instead of 12 of stored f_b.  Cells next to obstacles or walls read the
// stored field (their D3Q7 ghost-value gradient, k_body_force_near).  PER:
// every axis is periodic, so no source lies beyond a wall.  The near cells
// take a tenth of the kernel at a few per cent of the cells, bound by the
// instructions of 18 directions: their sources are the wrapped ones of the
// pull, a wall six bits of the cell against the direction's constant ones
// (instead of an index test and three wraps a direction), and a sphere's
// state comes as two 16-byte loads and one more (instead of nine).  Without
// PER the wall bits cost a register that spills at 48: 512^3 periodic 3.94 ms
// against 3.79 (3.89 before), 288 x 576 x 288 with walls 1.48 (1.56 before);
// FP16 256^3 444 -> 413 us, 96^3 55 -> 52 us.
template <class S, bool SLIP, bool FBPSI, bool EARLY, bool PER, class C = typename Store<S>::C>
__device__ __forceinline__ void lbm_cell(const Grid& g, const Streams<S>& P, const uint8_t* __restrict__ flags,
                                         const int32_t* __restrict__ owner, const DParticle* __restrict__ part,
                                         const float* __restrict__ partf, const C* __restrict__ fb, C ax, C ay,
                                         C az, const Trt<C>& R, int slip_faces, const FbPsi& fp, int x, int y,
                                         int z) {
    using St = Store<S>;
    const unsigned N = (unsigned)g.N;
    const int nx = g.nx, nxy = g.nx * g.ny;
    const int c = x + nx * (y + g.ny * z);
    const uint8_t fl = flags[c];
    // The pull sources x - e_q with every axis wrapped: in bounds for every
    // cell, and the true sources of all cells but the few next to an
    // obstacle or a wall.  EARLY: they are loaded before the cell's flags
    // arrive, so the two loads do not follow one another (obstacle cells
    // load and drop them, and cells next to an obstacle keep those of their
    // fluid neighbours, the same cells, and replace the others below);
    // otherwise each path loads what it needs after the flags (fewer live
    // registers, for the persistent batched kernel).  Same values either way.
    const int sx[3] = {(x == nx - 1 ? 0 : x + 1) - x, 0, (x == 0 ? nx - 1 : x - 1) - x};
    const int sy[3] = {((y == g.ny - 1 ? 0 : y + 1) - y) * nx, 0, ((y == 0 ? g.ny - 1 : y - 1) - y) * nx};
    const int sz[3] = {((z == g.nz - 1 ? 0 : z + 1) - z) * nxy, 0, ((z == 0 ? g.nz - 1 : z - 1) - z) * nxy};
    C f[19];
    auto pull = [&]() {
#pragma unroll
        for (int q = 0; q < 19; q++) {
            const int s_ = c + sx[1 + cx(q)] + sy[1 + cy(q)] + sz[1 + cz(q)];
            f[q] = St::ld(q, __ldg(P.src[q] + s_));
        }
    };
    if constexpr (EARLY) pull();
    if (fl & F_SOLID) return;  // obstacle cells are not updated

    C fx, fy, fz;  // body force (Sec. 5.6) plus the uniform acceleration
    if (!(fl & F_NEAR19)) {
        // all 18 pull sources are fluid cells inside the (periodic) domain
        if constexpr (FBPSI) {
            float f0, f1, f2;
            body_force_iso(load_psi19(fp.psi + c, sx, sy, sz), fp.Ex, fp.Ey, fp.Ez, fp.k2e, f0, f1, f2);
            fx = f0 + ax;
            fy = f1 + ay;
            fz = f2 + az;
        } else {
            fx = fb[c] + ax;
            fy = fb[N + c] + ay;
            fz = fb[2u * N + c] + az;
        }
        if constexpr (!EARLY) pull();
    } else {
        fx = fb[c] + ax;
        fy = fb[N + c] + ay;
        fz = fb[2u * N + c] + az;
        if constexpr (!EARLY) f[0] = St::ld(0, P.src[0][c]);
        // the non-periodic faces that the cell lies at, two bits an axis
        const unsigned wall =
            PER ? 0u
                : (g.per[0] ? 0u : (x == 0 ? 1u : 0u) | (x == nx - 1 ? 2u : 0u)) |
                      (g.per[1] ? 0u : (y == 0 ? 4u : 0u) | (y == g.ny - 1 ? 8u : 0u)) |
                      (g.per[2] ? 0u : (z == 0 ? 16u : 0u) | (z == g.nz - 1 ? 32u : 0u));
        unsigned hit = 0;  // FP64: directions whose source is an obstacle cell
        int o1 = -1;       // the first one's sphere
        int k0 = 0, k1 = 0, k2 = 0;
        bool many = false;
#pragma unroll
        for (int q = 1; q < 19; q++) {
            const int nb = c + sx[1 + cx(q)] + sy[1 + cy(q)] + sz[1 + cz(q)];
            const int o = owner[nb];
            if (!PER && (wall & crossed(q))) {
                if constexpr (SLIP) {
                    const WallSrc w = wall_source(g, slip_faces, owner, x, y, z, q, c);
                    f[q] = St::ld(q, P.src[w.q][w.cell]);
                } else {
                    f[q] = St::ld(opp(q), P.src[opp(q)][c]);  // resting no-slip wall: bounce back
                }
                continue;
            }
            if (o < 0) {  // a fluid source: the value pulled above
                if constexpr (!EARLY) f[q] = St::ld(q, P.src[q][nb]);
                continue;
            }
            // moving bounce-back (Eq. LBMMovWall): the population sent from x
            // towards the surface cell returns with 2 w_q rho_0 (c_q . u_s)/c_s^2
            if constexpr (sizeof(C) == 4) {
                // FP32 form: lever arm from the float copy of the particle
                const float4* p4 = reinterpret_cast<const float4*>(partf + 12 * o);
                const float4 pa = p4[0], pb = p4[1];
                const float pf[9] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w, partf[12 * o + 8]};
                float r[3] = {(float)x + 0.5f - (float)cx(q) - pf[0], (float)y + 0.5f - (float)cy(q) - pf[1],
                              (float)z + 0.5f - (float)cz(q) - pf[2]};
                const float Lw[3] = {(float)g.nx, (float)g.ny, (float)g.nz};
#pragma unroll
                for (int a = 0; a < 3; a++)
                    if (PER || g.per[a]) {
                        if (r[a] > 0.5f * Lw[a]) r[a] -= Lw[a];
                        if (r[a] < -0.5f * Lw[a]) r[a] += Lw[a];
                    }
                const float u0 = pf[3] + (pf[7] * r[2] - pf[8] * r[1]);
                const float u1 = pf[4] + (pf[8] * r[0] - pf[6] * r[2]);
                const float u2 = pf[5] + (pf[6] * r[1] - pf[7] * r[0]);
                const float cu = (float)cx(q) * u0 + (float)cy(q) * u1 + (float)cz(q) * u2;
                f[q] = St::ld(opp(q), P.src[opp(q)][c]) + (float)(6.0 * wq(q)) * cu;
            } else {
                f[q] = St::ld(opp(q), P.src[opp(q)][c]);
                many = many || (hit != 0u && o != o1);
                if (hit == 0u) {
                    o1 = o;
                    k0 = cx(q);
                    k1 = cy(q);
                    k2 = cz(q);
                }
                hit |= 1u << q;
            }
        }
        if constexpr (sizeof(C) == 8) {
            // u_s = V + Omega x (r - c_q) with r from the sphere's centre to
            // this fluid cell, and c_q . (Omega x c_q) = 0: so c_q . u_s =
            // c_q . U with one U = V + Omega x r for the cell, where the
            // sphere's image is the same for all its directions.  (A lever arm
            // for each direction is some 35 FP64 instructions, and a warp at a
            // surface has most of the 18 directions: 128^3 channel of 64
            // spheres 757 -> 622 us, 160 x 136 x 152 with 24 960 -> 900.)
            if (hit) {
                const DParticle& d = part[o1];
                double r[3] = {cell_disp(g, 0, wrap1(x - k0, g.nx), d.x[0]) + k0,
                               cell_disp(g, 1, wrap1(y - k1, g.ny), d.x[1]) + k1,
                               cell_disp(g, 2, wrap1(z - k2, g.nz), d.x[2]) + k2};
                const double U[3] = {d.v[0] + (d.w[1] * r[2] - d.w[2] * r[1]),
                                     d.v[1] + (d.w[2] * r[0] - d.w[0] * r[2]),
                                     d.v[2] + (d.w[0] * r[1] - d.w[1] * r[0])};
                // an obstacle cell within one cell of half the box away may be
                // the next image's: then, and next to two spheres, each
                // direction has its own lever arm
                const int n3[3] = {g.nx, g.ny, g.nz};
#pragma unroll
                for (int a = 0; a < 3; a++)
                    many = many || (g.per[a] && fabsf((float)r[a]) + 1.01f > 0.5f * (float)n3[a]);
                if (!many) {
#pragma unroll
                    for (int q = 1; q < 19; q++)
                        if ((hit >> q) & 1u) f[q] += (C)(6.0 * wq(q)) * dot_c(q, U);
                } else {
#pragma unroll
                    for (int q = 1; q < 19; q++) {
                        if (!((hit >> q) & 1u)) continue;
                        const int bx = wrap1(x - cx(q), g.nx), by = wrap1(y - cy(q), g.ny),
                                  bz = wrap1(z - cz(q), g.nz);
                        const DParticle& dq = part[owner[bx + g.nx * (by + g.ny * bz)]];
                        double us[3];
                        surface_velocity(g, dq.x, dq.v, dq.w, bx, by, bz, us);
                        f[q] += (C)(6.0 * wq(q)) * dot_c(q, us);
                    }
                }
            }
        }
    }

    auto put = [&](int q, C v) { P.dst[q][c] = St::st(q, v); };
    if constexpr (sizeof(C) == 4)
        collide_direct<C>(f, fx, fy, fz, R.lam_e, R.lam_o, put);
    else
        collide<C>(f, fx, fy, fz, R, put);
}

// One thread per cell; a block covers blockDim.x cells of blockDim.y rows
// (the shape is a parameter: es_params.lbm_block).
// (the reduced forms cap a thread at 48 registers, 1,280 threads per SM: with
// the pull loads issued ahead of the flag test, 40 registers spill and 64
// leave too few threads; both measured slower)
template <class S, bool SLIP, bool FBPSI, bool PER, class C = typename Store<S>::C>
__global__ void __launch_bounds__(256, sizeof(S) == 8 ? 3 : 5) k_lbm(Grid g, const Streams<S> P, const uint8_t* __restrict__ flags,
                                             const int32_t* __restrict__ owner, const DParticle* __restrict__ part,
                                             const float* __restrict__ partf, const C* __restrict__ fb, C ax, C ay,
                                             C az, const Trt<C> R, int slip_faces, FbPsi fp) {
    pdl_wait();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    lbm_cell<S, SLIP, FBPSI, true, PER>(g, P, flags, owner, part, partf, fb, ax, ay, az, R, slip_faces, fp, x, y, z);
}

// Several resident runs stepped by one persistent launch (es_lbm_step_batch):
// a work table of the runs' fields and parameters, passed by value, and a
// flat index of tiles of 32 cells x 4 rows over all runs (run r owns tiles
// tile0[r] .. tile0[r+1]-1).  Blocks of 128 threads stride over the tiles;
// each cell runs the same lbm_cell as k_lbm, so a run gives the same bits
// alone and in a batch.
constexpr int kBatchTileX = 32, kBatchTileY = 4;

template <class S>
struct BatchRun {
    using C = typename Store<S>::C;
    Grid g;
    Streams<S> P;
    const uint8_t* flags;
    const int32_t* owner;
    const DParticle* part;
    const float* partf;
    const C* fb;
    C ax, ay, az;
    Trt<C> R;
    FbPsi fp;
    int lazy;        // f_b from psi inside the stream-collide
    int tiles_x;     // tiles per row of tiles: ceil(nx / 32)
    int tiles_y;     // rows of tiles per plane: ceil(ny / 4)
    long long tile0; // first tile of the run
};

template <class S>
struct BatchTable {
    BatchRun<S> r[ES_LBM_BATCH_MAX];
    int n;
    long long ntiles;
};

template <class S>
__global__ void __launch_bounds__(kBatchTileX * kBatchTileY, sizeof(S) == 8 ? 6 : 8)
    k_lbm_batch(const __grid_constant__ BatchTable<S> T) {
    const int tx = threadIdx.x % kBatchTileX, ty = threadIdx.x / kBatchTileX;
    int r = 0;
    for (long long t = blockIdx.x; t < T.ntiles; t += gridDim.x) {
        while (r + 1 < T.n && T.r[r + 1].tile0 <= t) r++;
        const BatchRun<S>& R = T.r[r];
        const long long loc = t - R.tile0;
        const int bx = (int)(loc % R.tiles_x);
        const long long rest = loc / R.tiles_x;
        const int by = (int)(rest % R.tiles_y), z = (int)(rest / R.tiles_y);
        const int x = bx * kBatchTileX + tx, y = by * kBatchTileY + ty;
        if (x >= R.g.nx || y >= R.g.ny) continue;
        if constexpr (std::is_same<typename Store<S>::C, float>::value) {
            if (R.lazy) {
                lbm_cell<S, false, true, false, false>(R.g, R.P, R.flags, R.owner, R.part, R.partf, R.fb, R.ax, R.ay, R.az,
                                         R.R, 0, R.fp, x, y, z);
                continue;
            }
        }
        lbm_cell<S, false, false, false, false>(R.g, R.P, R.flags, R.owner, R.part, R.partf, R.fb, R.ax, R.ay, R.az, R.R, 0, R.fp, x, y, z);
    }
}

// Momentum exchange (Eq. LBMhydrodynForce): one block per sphere.  Each
// link x_F -> x_F + e_q into the sphere adds [2 f~_q(x_F) - 2 w_q (c_q . u_s)/c_s^2] c_q
// and the torque (x_s - X) x dF.  On small grids a few such blocks are all
// that runs, so their length is what counts, and a sphere's box holds twenty
// cells for every one with links.  The block therefore
//  * holds the rows of its box (one-cell halo included) as bit words, one for
//    the sphere's cells and one for fluid cells, built with a load and two
//    ballots a row;
//  * finds the cells with links a whole row at a time by shifts of those
//    words, and lists them (a prefix sum: in the order of their box index);
//  * then works on that list only.
// Boxes whose rows exceed 32 cells (R > 13) look the cells near the sphere's
// surface up in the fields (force_cells_fields).  Fixed order: deterministic.
constexpr int kForceChunk = 256;   // cells of a chunk (see k_forces_f32)
constexpr int kForceEach = 8;      // cells a thread looks up in the fields at a time
constexpr int kForceLinks = 4608;  // links held at once: at least one chunk's 18 x 256
constexpr int kForceSide = 32;     // longest row (halo included) of the bit words
constexpr int kForceChunks = (kForceSide - 2) * (kForceSide - 2) * (kForceSide - 2) / kForceChunk + 1;

// Components of the direction q, from two bits each.
__host__ __device__ constexpr unsigned long long dir_code(int a) {
    unsigned long long v = 0;
    for (int q = 0; q < 19; q++) v |= (unsigned long long)((a == 0 ? cx(q) : (a == 1 ? cy(q) : cz(q))) + 1) << (2 * q);
    return v;
}
__device__ __forceinline__ void dir_of(int q, int (&v)[3]) {
    constexpr unsigned long long X = dir_code(0), Y = dir_code(1), Z = dir_code(2);
    v[0] = (int)((X >> (2 * q)) & 3u) - 1;
    v[1] = (int)((Y >> (2 * q)) & 3u) - 1;
    v[2] = (int)((Z >> (2 * q)) & 3u) - 1;
}

// Local indices of a box cell from its linear index (x fastest).  Boxes of up
// to 2^20 cells divide by a multiplication: t / d = (t ceil(2^32 / d)) >> 32
// for t d < 2^32.
struct BoxIndex {
    int sx, sy, sxy;
    unsigned mx, mxy;
    bool quick;
    __device__ __forceinline__ BoxIndex(int sx_, int sy_, int n) : sx(sx_), sy(sy_), sxy(sx_ * sy_) {
        quick = n <= (1 << 20) && sxy < (1 << 11) && sx > 1;
        mx = (unsigned)((0x100000000ULL + sx - 1) / sx);
        mxy = (unsigned)((0x100000000ULL + sxy - 1) / sxy);
    }
    __device__ __forceinline__ void at(int t, int (&v)[3]) const {
        if (quick) {
            v[2] = (int)__umulhi((unsigned)t, mxy);
            const int r = t - v[2] * sxy;
            v[1] = (int)__umulhi((unsigned)r, mx);
            v[0] = r - v[1] * sx;
        } else {
            v[0] = t % sx;
            v[1] = (t / sx) % sy;
            v[2] = t / sxy;
        }
    }
};

// Exclusive prefix sum over the block (T threads), and its total.
template <int T>
__device__ __forceinline__ int block_excl(int v, int* s_warp, int& total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    const int w = lane < T / 32 ? s_warp[lane] : 0;
    total = __reduce_add_sync(0xffffffffu, w);
    const int before = __reduce_add_sync(0xffffffffu, lane < wid ? w : 0);
    __syncthreads();
    return before + incl - v;
}

// The links of a cell from the fields (boxes too large for the bit words).
__device__ __noinline__ unsigned force_links_fields(const Grid& g, const int32_t* __restrict__ owner,
                                                    const uint8_t* __restrict__ flags, int p, int x, int y, int z) {
    x = wrap_coord(x, g.nx);
    y = wrap_coord(y, g.ny);
    z = wrap_coord(z, g.nz);
    unsigned mask = 0;
    if (flags[x + g.nx * (y + g.ny * z)] & F_NEAR19) {
#pragma unroll
        for (int q = 1; q < 19; q++) {
            long long nb;
            if (neighbour(g, x, y, z, cx(q), cy(q), cz(q), nb) && owner[nb] == p) mask |= 1u << q;
        }
    }
    return mask;
}

// A sphere's box and the list of its cells with links.
struct ForceBox {
    int lo[3], n[3];
    int warp[32];
};

__device__ __forceinline__ void force_box(const Grid& g, const DParticle& P, ForceBox& B) {
    if (threadIdx.x < 3) {
        const int a = threadIdx.x;
        int l, h;
        axis_range(g, a, P.x[a], P.x[a], P.R, 1, l, h);
        B.lo[a] = l;
        B.n[a] = h - l + 1;
    }
    __syncthreads();
}

__device__ __forceinline__ bool force_by_rows(const ForceBox& B) {
    return B.n[0] + 2 <= kForceSide && B.n[1] + 2 <= kForceSide && B.n[2] + 2 <= kForceSide;
}

// The cells with links in s_near (box index) and s_mask (bit q: a link along
// q), by rows of bits; own, fluid: a word a row of the box with its halo.
// Returns their number.
template <int T>
__device__ __forceinline__ int force_cells(const Grid& g, const int32_t* __restrict__ owner, int p, ForceBox& B,
                                           const BoxIndex& bi, unsigned* own, unsigned* fluid, int* s_near,
                                           unsigned* s_mask) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int sx = B.n[0], sy = B.n[1], sz = B.n[2], ry = sy + 2, nr = ry * (sz + 2);
    // this lane's column, wrapped once
    const int gx0 = B.lo[0] - 1 + lane;
    const bool xin = lane < sx + 2 && (g.per[0] || (gx0 >= 0 && gx0 < g.nx));
    const int gx = xin ? wrap1(gx0, g.nx) : 0;
    int jz = wid / ry, jy = wid - jz * ry;
    for (int r0 = wid; r0 < nr; r0 += 4 * (T / 32)) {
        int o[4];
        bool in[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int y0 = B.lo[1] - 1 + jy, z0 = B.lo[2] - 1 + jz;
            in[u] = xin && r0 + u * (T / 32) < nr && (g.per[1] || (y0 >= 0 && y0 < g.ny)) &&
                    (g.per[2] || (z0 >= 0 && z0 < g.nz));
            o[u] = in[u] ? owner[gx + g.nx * (wrap1(y0, g.ny) + g.ny * wrap1(z0, g.nz))] : 0;
            for (jy += T / 32; jy >= ry; jy -= ry) jz++;
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const unsigned wo = __ballot_sync(0xffffffffu, in[u] && o[u] == p);
            const unsigned wf = __ballot_sync(0xffffffffu, in[u] && o[u] < 0);
            if (lane == 0 && r0 + u * (T / 32) < nr) {
                own[r0 + u * (T / 32)] = wo;
                fluid[r0 + u * (T / 32)] = wf;
            }
        }
    }
    __syncthreads();
    // rows of the box: cells with links, listed in the order of the box index
    const int rows = sy * sz, per = (rows + T - 1) / T;
    const unsigned inside = sx >= 31 ? 0x7ffffffeu : (((1u << sx) - 1u) << 1);
    auto any_of = [&](int r) {
        const int k = r / sy, at = (r - k * sy) + 1 + ry * (k + 1);
        unsigned m = 0;
        auto three = [&](int d) {
            const unsigned w = own[at + d];
            return w | (w << 1) | (w >> 1);
        };
        m = (own[at] << 1) | (own[at] >> 1);
        m |= three(-1) | three(1) | three(-ry) | three(ry);
        m |= own[at - 1 - ry] | own[at + 1 - ry] | own[at - 1 + ry] | own[at + 1 + ry];
        return m & fluid[at] & inside;
    };
    int cnt = 0;
    for (int u = 0; u < per; u++) {
        const int r = (int)threadIdx.x * per + u;
        if (r < rows) cnt += __popc(any_of(r));
    }
    int total;
    int at = block_excl<T>(cnt, B.warp, total);
    for (int u = 0; u < per; u++) {
        const int r = (int)threadIdx.x * per + u;
        if (r < rows)
            for (unsigned m = any_of(r); m; m &= m - 1u) s_near[at++] = r * sx + __ffs(m) - 2;  // (bit i + 1: cell i)
    }
    __syncthreads();
    for (int c = threadIdx.x; c < total; c += T) {
        int v[3];
        bi.at(s_near[c], v);
        const int w0 = v[1] + 1 + ry * (v[2] + 1), b = v[0] + 1;
        unsigned m = 0;
#pragma unroll
        for (int q = 1; q < 19; q++) m |= ((own[w0 + cy(q) + ry * cz(q)] >> (b + cx(q))) & 1u) << q;
        s_mask[c] = m;
    }
    __syncthreads();
    return total;
}

// The cells with links among the box's cells t0 .. t0 + kForceEach T - 1, from
// the fields, a thread a run of kForceEach of them.  A link runs from a fluid
// cell to a cell of p within sqrt 2, and p's cells are those within R of its
// centre at the last mapping, so only cells between R - 1 and R + 1.5 of that
// centre are looked up (FP32 distances; the bounds are far outside their
// rounding): a tenth of the box.  (One sphere R = 16 / R = 24: reduced forms
// 971 / 3,020 us looking at every cell 256 at a time, 311 / 878 so; FP64 1,128 /
// 3,410 and 326 / 809.)
template <int T>
__device__ __forceinline__ int force_cells_fields(const Grid& g, const int32_t* __restrict__ owner,
                                                  const uint8_t* __restrict__ flags, int p, ForceBox& B,
                                                  const BallF& ball, bool shell, float R, const BoxIndex& bi, int t0,
                                                  int n, int* s_near, unsigned* s_mask) {
    const float rin = R - 1.0f, rout = R + 1.5f, in2 = rin > 0.0f ? rin * rin : -1.0f, out2 = rout * rout;
    const int first = t0 + (int)threadIdx.x * kForceEach;
    unsigned m[kForceEach];
    int cnt = 0, v[3];
    bi.at(first < n ? first : 0, v);
#pragma unroll
    for (int u = 0; u < kForceEach; u++) {
        m[u] = 0;
        if (first + u < n) {
            const float d2 = shell ? ball.d2(v[0], v[1], v[2]) : in2;
            if (d2 >= in2 && d2 <= out2)
                m[u] = force_links_fields(g, owner, flags, p, B.lo[0] + v[0], B.lo[1] + v[1], B.lo[2] + v[2]);
        }
        cnt += m[u] != 0;
        if (++v[0] == B.n[0]) {
            v[0] = 0;
            if (++v[1] == B.n[1]) {
                v[1] = 0;
                v[2]++;
            }
        }
    }
    int total;
    int at = block_excl<T>(cnt, B.warp, total);
#pragma unroll
    for (int u = 0; u < kForceEach; u++)
        if (m[u]) {
            s_near[at] = first + u;
            s_mask[at++] = m[u];
        }
    __syncthreads();
    return total;
}

// The mapped centre's ball relative to the box, for that (every thread calls).
__device__ __forceinline__ bool force_ball(const Grid& g, const double* __restrict__ X, double R, const ForceBox& B,
                                           BallF& ball) {
    const int hi[3] = {B.lo[0] + B.n[0] - 1, B.lo[1] + B.n[1] - 1, B.lo[2] + B.n[2] - 1};
    ball.init_by_axis(g, X, R, B.lo, hi);
    __syncthreads();
    return ball.all_ok();
}

// Half the force and torque of the links m of cell (x, y, z), link by link.
__device__ __noinline__ void force_links_each(const Grid& g, const DParticle& P, unsigned m, int x, int y, int z,
                                              const double* __restrict__ src, size_t ps, double (&acc)[6]) {
    const int c = x + g.nx * (y + g.ny * z);
    for (; m; m &= m - 1u) {
        const int q = __ffs(m) - 1;
        int v[3];
        dir_of(q, v);
        const int bx = wrap_coord(x + v[0], g.nx), by = wrap_coord(y + v[1], g.ny), bz = wrap_coord(z + v[2], g.nz);
        const double r0 = cell_disp(g, 0, bx, P.x[0]), r1 = cell_disp(g, 1, by, P.x[1]), r2 = cell_disp(g, 2, bz, P.x[2]);
        double us[3];
        surface_velocity(g, P.x, P.v, P.w, bx, by, bz, us);
        const double w = (q <= 3 || (q >= 10 && q <= 12)) ? 1.0 / 18.0 : 1.0 / 36.0;
        const double mq = src[q * ps + c] - 3.0 * w * (v[0] * us[0] + v[1] * us[1] + v[2] * us[2]);
        const double d0 = mq * v[0], d1 = mq * v[1], d2 = mq * v[2];
        acc[0] += d0;
        acc[1] += d1;
        acc[2] += d2;
        acc[3] += r1 * d2 - r2 * d1;
        acc[4] += r2 * d0 - r0 * d2;
        acc[5] += r0 * d1 - r1 * d0;
    }
}

// FP64 form.  The FP64 pipe (2 operations a clock and SM) bounds it, so a
// cell's links share what they can: u_s . c_q = u_F . c_q with u_F = V + W x
// r_F, since x_s = x_F + c_q and (W x c_q) . c_q = 0, and the torques add up to
// r_F x sum m_q c_q, since c_q x c_q = 0.  A warp has links along all 18
// directions, so a cell takes them by pairs without a branch: with b = 1 where
// there is a link (f = 0 where not), m_q - m_-q = 2 [f_q - f_-q - 3 w_q (b_q +
// b_-q) u_F . c_q]; 39 instructions for the 18 instead of 78.  The block's sums
// exchange halves of the six components instead of adding all six at each of
// five steps (8 instructions a warp, not 30), in the warps that have cells.
// (A sphere R = 4 / 64 spheres R = 6: 62 / 133 us with a lever arm a link, 32
// / 48 link by link, 23 / 37 now.)
template <int T>
__global__ void __launch_bounds__(T, 1) k_forces(Grid g, const DParticle* __restrict__ part,
                                                 const int32_t* __restrict__ owner, const uint8_t* __restrict__ flags,
                                                 const double* __restrict__ src, double Ex, double Ey, double Ez,
                                                 const double* __restrict__ mapped, double* F, double* T_out,
                                                 int cells) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ ForceBox B;
    __shared__ BallF ball;
    __shared__ double sh[6][32];
    unsigned* own = (unsigned*)dyn;
    unsigned* fluid = own + kForceSide * kForceSide;
    int* s_near = (int*)(fluid + kForceSide * kForceSide);
    unsigned* s_mask = (unsigned*)(s_near + cells);
    const int p = blockIdx.x;
    pdl_wait();
    force_box(g, part[p], B);
    const int n = B.n[0] * B.n[1] * B.n[2];
    const BoxIndex bi(B.n[0], B.n[1], n);
    const DParticle& P = part[p];
    const double X[3] = {P.x[0], P.x[1], P.x[2]}, V[3] = {P.v[0], P.v[1], P.v[2]}, Wv[3] = {P.w[0], P.w[1], P.w[2]};
    const size_t ps = (size_t)g.ps;
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    int active = 0;  // warps that have had cells
    auto consume = [&](int total) {
        const int w = (total + 31) / 32;
        active = w > active ? (w < T / 32 ? w : T / 32) : active;
        for (int i = threadIdx.x; i < total; i += T) {
            int v[3];
            bi.at(s_near[i], v);
            const unsigned m = s_mask[i];
            const int x = wrap_coord(B.lo[0] + v[0], g.nx), y = wrap_coord(B.lo[1] + v[1], g.ny),
                      z = wrap_coord(B.lo[2] + v[2], g.nz);
            const int c = x + g.nx * (y + g.ny * z);
            const double r0 = cell_disp(g, 0, x, X[0]), r1 = cell_disp(g, 1, y, X[1]), r2 = cell_disp(g, 2, z, X[2]);
            const double u[3] = {V[0] + (Wv[1] * r2 - Wv[2] * r1), V[1] + (Wv[2] * r0 - Wv[0] * r2),
                                 V[2] + (Wv[0] * r1 - Wv[1] * r0)};
            // a sphere that moved since its mapping may have a fluid cell past
            // half a periodic axis whose surface cells are not: then each
            // link has its own lever arm, at its surface cell's nearest image
            const double r3[3] = {r0, r1, r2};
            const int n3[3] = {g.nx, g.ny, g.nz};
            bool past = false;
#pragma unroll
            for (int a = 0; a < 3; a++) past |= g.per[a] && fabsf((float)r3[a]) + 1.01f > 0.5f * (float)n3[a];
            if (past) {
                force_links_each(g, P, m, x, y, z, src, ps, acc);
                continue;
            }
            double d[3] = {0.0, 0.0, 0.0};  // half the sum of m_q c_q
            // three pairs of populations in flight at a time
#pragma unroll
            for (int q0 = 1; q0 <= 9; q0 += 3) {
                double f[3], h[3];
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    f[j] = ((m >> (q0 + j)) & 1u) ? src[(q0 + j) * ps + c] : 0.0;
                    h[j] = ((m >> (q0 + j + 9)) & 1u) ? src[(q0 + j + 9) * ps + c] : 0.0;
                }
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    const int q = q0 + j;
                    const unsigned b0 = (m >> q) & 1u, b1 = (m >> (q + 9)) & 1u;
                    const double k = (b0 & b1) ? -6.0 * wq(q) : ((b0 | b1) ? -3.0 * wq(q) : 0.0);
                    const double mq = (f[j] - h[j]) + k * dot_c(q, u);
                    if (cx(q)) d[0] += cx(q) > 0 ? mq : -mq;
                    if (cy(q)) d[1] += cy(q) > 0 ? mq : -mq;
                    if (cz(q)) d[2] += cz(q) > 0 ? mq : -mq;
                }
            }
            acc[0] += d[0];
            acc[1] += d[1];
            acc[2] += d[2];
            acc[3] += r1 * d[2] - r2 * d[1];
            acc[4] += r2 * d[0] - r0 * d[2];
            acc[5] += r0 * d[1] - r1 * d[0];
        }
    };
    if (force_by_rows(B)) {
        consume(force_cells<T>(g, owner, p, B, bi, own, fluid, s_near, s_mask));
    } else {
        const bool shell = force_ball(g, mapped + 9 * p, P.R, B, ball);
        for (int t0 = 0; t0 < n; t0 += kForceEach * T) {
            consume(force_cells_fields<T>(g, owner, flags, p, B, ball, shell, (float)P.R, bi, t0, n, s_near, s_mask));
            __syncthreads();
        }
    }
    // block sums in a fixed order: the warps that had cells (half a warp keeps
    // three components, a quarter two of four, ...), then one thread per
    // component
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < active) {
        const bool up = lane & 16, up2 = lane & 8, up3 = lane & 4;
        double a3[4];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const double mine = up ? acc[k + 3] : acc[k], other = up ? acc[k] : acc[k + 3];
            a3[k] = mine + __shfl_xor_sync(0xffffffffu, other, 16);
        }
        a3[3] = 0.0;
        double a2[2];
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const double mine = up2 ? a3[k + 2] : a3[k], other = up2 ? a3[k] : a3[k + 2];
            a2[k] = mine + __shfl_xor_sync(0xffffffffu, other, 8);
        }
        double a1 = (up3 ? a2[1] : a2[0]) + __shfl_xor_sync(0xffffffffu, up3 ? a2[0] : a2[1], 4);
        a1 += __shfl_xor_sync(0xffffffffu, a1, 2);
        a1 += __shfl_xor_sync(0xffffffffu, a1, 1);
        const int k = (up2 ? 2 : 0) + (up3 ? 1 : 0);
        if ((lane & 3) == 0 && k < 3) sh[(up ? 3 : 0) + k][wid] = a1;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        double s = 0.0;
        for (int w = 0; w < active; w++) s += sh[k][w];
        s *= 2.0;
        const double E[3] = {Ex, Ey, Ez};
        if (k < 3)
            F[3 * p + k] = s + P.qeff * E[k];  // F_C = q E_ext (Sec. 5.6)
        else
            T_out[3 * p + k - 3] = s;
    }
}

// Momentum exchange of the reduced forms (float or FP16 populations, stored
// as deviations f - w_q).  Same links and sums as k_forces, arranged so that
// no FP64 arithmetic runs per link (GB300's FP64 rate is a small fraction
// of its FP32 rate).  With f~ = w_q + dev the link term is
// [2 w_q + m'] c_q, m' = 2 dev - 6 w_q (c_q . u_s):
//  * the m' part (small) is formed by all threads, one link each, with lever
//    arms in FP32, then summed in FP32 by 256 of them -- link i of a chunk of
//    256 box cells by thread i mod 256, chunk after chunk -- and over the block
//    in float-float;
//  * the 2 w_q part is summed exactly in integers: for each direction the
//    number of links and the sums of their surface cells' coordinates (relative
//    to the box, minimum image), a vote and a warp sum of the packed three a
//    direction, from which sum 2 w_q c_q and sum 2 w_q (x_s - X) x c_q follow in
//    FP64 at the end, direction by direction.
// (2,880 spheres R = 5 / 64 spheres R = 6: 277 / 83 us with an owner tile, a
// lookup a neighbour where it did not fit and four shared-memory atomics a link;
// 238 / 27 now.  The constant part as six integers a cell instead of a
// direction's sums is 221 / 25, but rounds differently at the end.)
template <class S, int T>
__global__ void __launch_bounds__(T, T == 1024 ? 1 : 3)
    k_forces_f32(Grid g, const DParticle* __restrict__ part, const int32_t* __restrict__ owner,
                 const uint8_t* __restrict__ flags, const S* __restrict__ src, double Ex, double Ey, double Ez,
                 const double* __restrict__ mapped, double* F, double* T_out, int cells) {
    using St = Store<S>;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ ForceBox B;
    __shared__ BallF ball;
    __shared__ float s_X[3], s_V[3], s_W[3];
    __shared__ double s_off[3], s_qeff;
    __shared__ int s_dir[19][4], s_first[kForceChunks], s_count[kForceChunks];
    __shared__ double s_term[19][6];
    __shared__ float s_red[kForceChunk / 32][12];
    unsigned* own = (unsigned*)dyn;
    unsigned* fluid = own + kForceSide * kForceSide;
    int* s_near = (int*)(fluid + kForceSide * kForceSide);
    unsigned* s_mask = (unsigned*)(s_near + cells);
    int* s_link = (int*)(s_mask + cells);         // cell of the list | q << 16
    float* s_m = (float*)(s_link + kForceLinks);  // its m'
    const int p = blockIdx.x;
    pdl_wait();
    force_box(g, part[p], B);
    if (threadIdx.x < 3) {
        const DParticle& P = part[p];
        const int a = threadIdx.x;
        // centre relative to the box origin's cell centre: r = i - s_X for
        // the cell with local index i (exact to FP32 rounding of s_X)
        const double off = (double)B.lo[a] + 0.5 - P.x[a];
        s_off[a] = off;
        s_X[a] = (float)(-off);
        s_V[a] = (float)P.v[a];
        s_W[a] = (float)P.w[a];
    }
    if (threadIdx.x == 32) s_qeff = part[p].qeff;
    if (threadIdx.x < 4 * 19) s_dir[threadIdx.x / 4][threadIdx.x % 4] = 0;
    __syncthreads();
    const int n = B.n[0] * B.n[1] * B.n[2];
    const BoxIndex bi(B.n[0], B.n[1], n);
    const float Xr[3] = {s_X[0], s_X[1], s_X[2]}, V[3] = {s_V[0], s_V[1], s_V[2]}, W[3] = {s_W[0], s_W[1], s_W[2]};
    const size_t ps = (size_t)g.ps;
    // a box index's minimum image (a periodic box may span the whole axis)
    auto image = [&](int u, int a) {
        const int L = a == 0 ? g.nx : (a == 1 ? g.ny : g.nz);
        if (g.per[a]) {
            if ((float)u - Xr[a] > 0.5f * (float)L) u -= L;
            if ((float)u - Xr[a] < -0.5f * (float)L) u += L;
        }
        return u;
    };
    float acc[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    // lane q of every warp: number of links along q, and the sums of their
    // surface cells' coordinates
    int nq = 0, sq[3] = {0, 0, 0};
    const int lane = threadIdx.x & 31;
    // Rows of bit words whose cells are their own nearest images: box
    // coordinates below 32, so a warp's sums of the three fit one word.
    bool packed = force_by_rows(B);
#pragma unroll
    for (int a = 0; a < 3; a++) packed &= !g.per[a] || B.n[a] + 4 <= gdim(g, a);
    // The listed cells' links: chunk of a cell: (box index - t0) / 256, nch chunks.
    auto consume = [&](int total, int t0, int nch) {
        for (int c = threadIdx.x; c < nch; c += T) s_count[c] = 0;
        __syncthreads();
        const int per = (total + T - 1) / T;
        int cnt = 0;
        for (int u = 0; u < per; u++) {
            const int c = (int)threadIdx.x * per + u;
            const bool on = c < total;
            if (!__any_sync(0xffffffffu, on)) break;
            const unsigned m = on ? s_mask[c] : 0u;
            int v[3] = {0, 0, 0};
            if (on) {
                const int t = s_near[c];
                cnt += __popc(m);
                atomicAdd(&s_count[(t - t0) / kForceChunk], __popc(m));
                bi.at(t, v);
            }
            const unsigned place = (unsigned)v[0] | ((unsigned)v[1] << 10) | ((unsigned)v[2] << 20);
            if (packed) {
#pragma unroll 6
                for (int q = 1; q < 19; q++) {
                    const bool b = (m >> q) & 1u;
                    const int n = __popc(__ballot_sync(0xffffffffu, b));
                    const unsigned w = __reduce_add_sync(0xffffffffu, b ? place : 0u);
                    if (lane == q) {
                        int d[3];
                        dir_of(q, d);
                        nq += n;
                        sq[0] += (int)(w & 1023u) + n * d[0];
                        sq[1] += (int)((w >> 10) & 1023u) + n * d[1];
                        sq[2] += (int)(w >> 20) + n * d[2];
                    }
                }
            } else {
#pragma unroll 1
                for (int q = 1; q < 19; q++) {
                    const bool b = (m >> q) & 1u;
                    const int n = __popc(__ballot_sync(0xffffffffu, b));
                    int d[3];
                    dir_of(q, d);
#pragma unroll
                    for (int a = 0; a < 3; a++) {
                        const int w = __reduce_add_sync(0xffffffffu, b ? image(v[a] + d[a], a) : 0);
                        if (lane == q) sq[a] += w;
                    }
                    if (lane == q) nq += n;
                }
            }
        }
        int nlinks;
        const int base = block_excl<T>(cnt, B.warp, nlinks);
        {
            int at = base;
            for (int u = 0; u < per; u++) {
                const int c = (int)threadIdx.x * per + u;
                if (c >= total) break;
                const int ch = (s_near[c] - t0) / kForceChunk;
                if (c == 0 || (s_near[c - 1] - t0) / kForceChunk != ch) s_first[ch] = at;
                at += __popc(s_mask[c]);
            }
        }
        __syncthreads();
        // as many chunks at a time as the link list holds (nearly always all)
        for (int k0 = 0, done = 0; k0 < nch;) {
            int k1 = k0, held = 0;
            if (nlinks - done <= kForceLinks) {
                k1 = nch;
                held = nlinks - done;
            } else {
                while (k1 < nch && held + s_count[k1] <= kForceLinks) held += s_count[k1++];
            }
            int at = base;
            for (int u = 0; u < per; u++) {
                const int c = (int)threadIdx.x * per + u;
                if (c >= total) break;
                const int ch = (s_near[c] - t0) / kForceChunk;
                unsigned m = s_mask[c];
                if (ch < k0 || ch >= k1) {
                    at += __popc(m);
                    continue;
                }
                for (; m; m &= m - 1u) s_link[at++ - done] = c | ((__ffs(m) - 1) << 16);
            }
            __syncthreads();
            for (int i = threadIdx.x; i < held; i += T) {
                const int link = s_link[i], q = link >> 16;
                int li[3], qv[3];
                bi.at(s_near[link & 0xFFFF], li);
                dir_of(q, qv);
                const int cc = wrap1(B.lo[0] + li[0], g.nx) +
                               g.nx * (wrap1(B.lo[1] + li[1], g.ny) + g.ny * wrap1(B.lo[2] + li[2], g.nz));
                const S f = src[q * ps + cc];
                float r[3];
#pragma unroll
                for (int a = 0; a < 3; a++) r[a] = (float)image(li[a] + qv[a], a) - Xr[a];
                const float us0 = V[0] + (W[1] * r[2] - W[2] * r[1]);
                const float us1 = V[1] + (W[2] * r[0] - W[0] * r[2]);
                const float us2 = V[2] + (W[0] * r[1] - W[1] * r[0]);
                const float cu = (float)qv[0] * us0 + (float)qv[1] * us1 + (float)qv[2] * us2;
                const float w = (q <= 3 || (q >= 10 && q <= 12)) ? 1.0f / 18.0f : 1.0f / 36.0f;
                float dev;  // f~ - w_q
                if constexpr (std::is_same<S, __half>::value)
                    dev = __half2float(f) * (w * (float)(1.0 / kHalfScale));  // (Store<__half>::ld in FP32)
                else
                    dev = St::ld(q, f);
                s_m[i] = 2.0f * dev - 6.0f * w * cu;
            }
            __syncthreads();
            if (threadIdx.x < kForceChunk)
                for (int ch = k0; ch < k1; ch++) {
                    const int nl = s_count[ch];
                    if (nl == 0) continue;
                    const int first = s_first[ch] - done;
                    for (int i = threadIdx.x; i < nl; i += kForceChunk) {
                        const int link = s_link[first + i];
                        const float m = s_m[first + i];
                        int li[3], qv[3];
                        bi.at(s_near[link & 0xFFFF], li);
                        dir_of(link >> 16, qv);
                        float r[3];
#pragma unroll
                        for (int a = 0; a < 3; a++) r[a] = (float)image(li[a] + qv[a], a) - Xr[a];
                        const float d0 = m * (float)qv[0], d1 = m * (float)qv[1], d2 = m * (float)qv[2];
                        acc[0] += d0;
                        acc[1] += d1;
                        acc[2] += d2;
                        acc[3] += r[1] * d2 - r[2] * d1;
                        acc[4] += r[2] * d0 - r[0] * d2;
                        acc[5] += r[0] * d1 - r[1] * d0;
                    }
                }
            __syncthreads();
            done += held;
            k0 = k1;
        }
    };
    if (force_by_rows(B)) {
        const int total = force_cells<T>(g, owner, p, B, bi, own, fluid, s_near, s_mask);
        consume(total, 0, (n + kForceChunk - 1) / kForceChunk);
    } else {
        const float R = (float)part[p].R;
        const bool shell = force_ball(g, mapped + 9 * p, part[p].R, B, ball);
        for (int t0 = 0; t0 < n; t0 += kForceEach * T)
            consume(force_cells_fields<T>(g, owner, flags, p, B, ball, shell, R, bi, t0, n, s_near, s_mask), t0,
                    kForceEach * T / kForceChunk);
    }
    // block sum of the six FP32 partials in float-float (fixed order)
    if (threadIdx.x < kForceChunk) {
        ff v[6];
#pragma unroll
        for (int k = 0; k < 6; k++) v[k] = {acc[k], 0.0f};
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 6; k++) {
                const ff u = {__shfl_down_sync(0xffffffffu, v[k].hi, o), __shfl_down_sync(0xffffffffu, v[k].lo, o)};
                v[k] = ff_add(v[k], u);
            }
        if ((threadIdx.x & 31) == 0)
#pragma unroll
            for (int k = 0; k < 6; k++) {
                s_red[threadIdx.x >> 5][2 * k] = v[k].hi;
                s_red[threadIdx.x >> 5][2 * k + 1] = v[k].lo;
            }
    }
    if (nq != 0) {
        atomicAdd(&s_dir[lane][0], nq);
#pragma unroll
        for (int a = 0; a < 3; a++) atomicAdd(&s_dir[lane][1 + a], sq[a]);
    }
    __syncthreads();
    // a direction's terms, a thread each: 2 w_q times its links (a force), and
    // the sum of (x_s - X) x c_q (a torque), x_s - X = the sums + links (lo + 1/2 - X)
    if (threadIdx.x < 6 * 18) {
        const int q = 1 + threadIdx.x / 6, k = threadIdx.x % 6, c = k % 3, d = (c + 1) % 3, e = (c + 2) % 3;
        int v[3];
        dir_of(q, v);
        auto sign = [&](int a, double x) {
            const int s = a == 0 ? v[0] : (a == 1 ? v[1] : v[2]);
            return s == 0 ? 0.0 : (s > 0 ? x : -x);
        };
        const double n = (double)s_dir[q][0], w2 = (q <= 3 || (q >= 10 && q <= 12)) ? 2.0 / 18.0 : 2.0 / 36.0;
        double t;
        if (k < 3) {
            t = sign(c, __dmul_rn(w2, n));
        } else {
            const double rd = __fma_rn(n, s_off[d], (double)s_dir[q][1 + d]),
                         re = __fma_rn(n, s_off[e], (double)s_dir[q][1 + e]);
            t = __dadd_rn(sign(e, rd), -sign(d, re));
        }
        s_term[q][k] = t;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        ff a = {s_red[0][2 * k], s_red[0][2 * k + 1]};
        for (int w = 1; w < kForceChunk / 32; w++) a = ff_add(a, ff{s_red[w][2 * k], s_red[w][2 * k + 1]});
        double sum = (double)a.hi + (double)a.lo;
        // (a force adds its terms, rounded; a torque takes 2 w_q with the addition)
#pragma unroll
        for (int q = 1; q < 19; q++)
            sum = __fma_rn(k < 3 ? 1.0 : 2.0 * wq(q), s_term[q][k], sum);
        if (k < 3)
            F[3 * p + k] = sum + s_qeff * (k == 0 ? Ex : (k == 1 ? Ey : Ez));  // F_C = q E_ext (Sec. 5.6)
        else
            T_out[3 * p + k - 3] = sum;
    }
}

// Semi-implicit Euler, dt = 1 (the integrator is a reading: the paper
// leaves it to the pe engine).
// A thread an axis of a sphere (its chain of FP64 operations is the kernel's
// time).  Keeps the float copy that the reduced forms' stream-collide reads.
__global__ void k_advance(int np, DParticle* part, const double* F, const double* T, int px, int py, int pz,
                          double Lx, double Ly, double Lz, float* __restrict__ pf) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (t >= 3 * np) return;
    const int p = t / 3, a = t - 3 * p;
    DParticle& P = part[p];
    const bool per = a == 0 ? px : (a == 1 ? py : pz);
    const double L = a == 0 ? Lx : (a == 1 ? Ly : Lz);
    const double w = P.w[a] + T[t] / P.inertia, v = P.v[a] + F[t] / P.mass;
    double x = P.x[a] + v;
    if (per) {
        if (x >= L) x -= L;
        if (x < 0.0) x += L;
    }
    P.v[a] = v;
    P.x[a] = x;
    P.w[a] = w;
    if (pf) {
        pf[12 * p + a] = (float)x;
        pf[12 * p + 3 + a] = (float)v;
        pf[12 * p + 6 + a] = (float)w;
    }
}

template <class S>
__global__ void k_fill_rest(int N, size_t ps, S* a, S* b) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int q = blockIdx.y;
    if (i >= N) return;
    const S v = Store<S>::rest(q);
    a[q * ps + i] = v;
    b[q * ps + i] = v;
}

// PDFs are exchanged densely (19 x N doubles) and stored with stride ps.
template <class S>
__global__ void k_get_pdf(long long N, long long ps, const S* src, double* dst) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 19 * N) return;
    int q = (int)(i / N);
    dst[i] = Store<S>::to_f(q, src[(long long)q * ps + (i - (long long)q * N)]);
}

template <class S>
__global__ void k_set_pdf(long long N, long long ps, const double* src, S* dst) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 19 * N) return;
    int q = (int)(i / N);
    dst[(long long)q * ps + (i - (long long)q * N)] = Store<S>::from_f(q, src[i]);
}

// Density or velocity of the FP64 form: rho = sum f, u = sum c f - f_b / 2
// (the collision keeps rho and adds exactly f_b).
template <bool RHO>
__global__ void __launch_bounds__(256) k_moments(long long N, long long ps, const double* __restrict__ f,
                                                 const double* __restrict__ fb, double ax, double ay, double az,
                                                 double* __restrict__ out) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    double r = 0.0, j0 = 0.0, j1 = 0.0, j2 = 0.0;
#pragma unroll
    for (int q = 0; q < 19; q++) {
        if (!RHO && q == 0) continue;
        const double v = f[(long long)q * ps + c];
        if (RHO) {
            r += v;
            continue;
        }
        if (cx(q)) j0 += cx(q) > 0 ? v : -v;
        if (cy(q)) j1 += cy(q) > 0 ? v : -v;
        if (cz(q)) j2 += cz(q) > 0 ? v : -v;
    }
    if (RHO) {
        out[c] = r;
    } else {
        out[c] = j0 - 0.5 * (fb[c] + ax);
        out[N + c] = j1 - 0.5 * (fb[N + c] + ay);
        out[2 * N + c] = j2 - 0.5 * (fb[2 * N + c] + az);
    }
}

// Density or velocity of the reduced forms.  The stored deviations are
// summed in float-float (TwoSum, about 48 bits) and widened to FP64 once per
// value: summed in FP64, the 100 FP64 operations a cell bound the kernel at
// 1/64 of the FP32 rate (density, velocity and potential of a 320^3 MIXED32
// state: 13.5 ms, in float-float 1.21 ms, 0.49 of the copy rate).  The
// deviations carry no
// w_q, so the sums hold more bits of the velocity than FP64 sums of
// w_q + dev do.  FP16 storage: the axis and the diagonal streams are summed
// apart and take their weight as a float-float product.  FBPSI: the body
// force of an interior cell is formed from psi as the stream-collide forms
// it (cells next to obstacles read the stored field, obstacle cells have
// none), so the whole field is neither stored nor read back.
//
// Sums that are not finite (a diverged state) are formed again in FP64: TwoSum
// makes NaN of an infinity.
struct Accel3 {
    ff a[3];  // - accel / 2
};

// Density or velocity of cell c in FP64; h: f_b plus the acceleration, halved.
template <class S, bool RHO>
__device__ __noinline__ void moments_fp64(const S* __restrict__ f, size_t ps, size_t N, int c, double h0, double h1,
                                          double h2, double* __restrict__ out) {
    double r = 0.0, j[3] = {0.0, 0.0, 0.0};
    for (int q = 0; q < 19; q++) {
        const double v = Store<S>::to_f(q, f[q * ps + c]);
        r += v;
        j[0] += cx(q) * v;
        j[1] += cy(q) * v;
        j[2] += cz(q) * v;
    }
    if (RHO) {
        out[c] = r;
    } else {
        out[c] = j[0] - h0;
        out[N + c] = j[1] - h1;
        out[2 * N + c] = j[2] - h2;
    }
}

template <class S, bool RHO, bool FBPSI>
__global__ void __launch_bounds__(256) k_moments_ff(Grid g, const S* __restrict__ f, const float* __restrict__ fb,
                                                    const uint8_t* __restrict__ flags, FbPsi fp, Accel3 acc,
                                                    double* __restrict__ out) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const int c = x + g.nx * (y + g.ny * z);
    constexpr bool kHalf = sizeof(S) == 2;
    // the weights of FP16 storage: dev = h w_q / 2^12
    constexpr float wa = (float)(1.0 / 18.0 / kHalfScale), wa2 = (float)(1.0 / 18.0 / kHalfScale - (double)wa);
    constexpr float wd = 0.5f * wa, wd2 = 0.5f * wa2;
    auto ld = [&](int q) -> float { return (float)__ldg(f + (size_t)q * g.ps + c); };
    if constexpr (RHO) {
        ff_acc s{0.0f, 0.0f}, d{0.0f, 0.0f};
#pragma unroll
        for (int q = 1; q < 19; q++) {
            if (kHalf && !(q <= 3 || (q >= 10 && q <= 12)))
                d.add(ld(q), 0.0f);
            else
                s.add(ld(q), 0.0f);
        }
        ff v;
        if constexpr (kHalf) {
            s.add(6.0f * ld(0), 0.0f);  // (w_0 = 6 w_1; an 11-bit value times 6 is exact)
            v = ff_add(ff_mul(s.value(), {wa, wa2}), ff_mul(d.value(), {wd, wd2}));
        } else {
            s.add(ld(0), 0.0f);
            v = s.value();
        }
        out[c] = 1.0 + widen(v);
        const float t = __fadd_rn(v.hi, v.lo);
        if (!(__fsub_rn(t, t) == 0.0f)) moments_fp64<S, true>(f, g.ps, 0, c, 0.0, 0.0, 0.0, out);
    } else {
        ff_acc s[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, d[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll
        for (int q = 1; q < 19; q++) {
            const float v = ld(q);
            const int cq[3] = {cx(q), cy(q), cz(q)};
#pragma unroll
            for (int a = 0; a < 3; a++)
                if (cq[a]) {
                    if (kHalf && !(q <= 3 || (q >= 10 && q <= 12)))
                        d[a].add(cq[a] > 0 ? v : -v, 0.0f);
                    else
                        s[a].add(cq[a] > 0 ? v : -v, 0.0f);
                }
        }
        const size_t N = (size_t)g.N;
        float b[3];
        bool stored = true, bad = false;
        if constexpr (FBPSI) {
            const uint8_t fl = flags[c];
            stored = (fl & (F_SOLID | F_NEAR19)) == F_NEAR19;
            b[0] = b[1] = b[2] = 0.0f;
            if (!(fl & (F_SOLID | F_NEAR19))) {
                const int nx = g.nx, nxy = g.nx * g.ny;
                const int sx[3] = {(x == nx - 1 ? 0 : x + 1) - x, 0, (x == 0 ? nx - 1 : x - 1) - x};
                const int sy[3] = {((y == g.ny - 1 ? 0 : y + 1) - y) * nx, 0, ((y == 0 ? g.ny - 1 : y - 1) - y) * nx};
                const int sz[3] = {((z == g.nz - 1 ? 0 : z + 1) - z) * nxy, 0, ((z == 0 ? g.nz - 1 : z - 1) - z) * nxy};
                body_force_iso(load_psi19(fp.psi + c, sx, sy, sz), fp.Ex, fp.Ey, fp.Ez, fp.k2e, b[0], b[1], b[2]);
            }
        }
        if (stored) {
#pragma unroll
            for (int a = 0; a < 3; a++) b[a] = fb[a * N + c];
        }
#pragma unroll
        for (int a = 0; a < 3; a++) {
            ff v;
            if constexpr (kHalf)
                v = ff_add(ff_mul(s[a].value(), {wa, wa2}), ff_mul(d[a].value(), {wd, wd2}));
            else
                v = s[a].value();
            v = ff_add(ff_add_f(v, -0.5f * b[a]), acc.a[a]);
            out[a * N + c] = widen(v);
            const float t = __fadd_rn(v.hi, v.lo);
            bad |= !(__fsub_rn(t, t) == 0.0f);
        }
        if (bad)
            moments_fp64<S, false>(f, g.ps, N, c, 0.5 * b[0] - widen(acc.a[0]), 0.5 * b[1] - widen(acc.a[1]),
                                   0.5 * b[2] - widen(acc.a[2]), out);
    }
}

template <class S>
__global__ void k_copy_fb(long long n, const S* a, double* b) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (double)a[i];
}

template <class S>
__global__ void k_load_fb(long long n, const double* a, S* b) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (S)a[i];
}

template <class S, class C = typename Store<S>::C>
__global__ void k_gather(int which, long long N, long long ps, const long long* idx, int n, const S* cur, const S* last,
                         const C* fb, const double* psi, const float* psi_hi, const float* psi_lo,
                         const int32_t* owner, const uint8_t* flags, double ax, double ay, double az, double* out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    long long c = idx[i];
    switch (which) {
    case ES_FIELD_PSI: out[i] = psi ? psi[c] : (double)psi_hi[c] + (double)psi_lo[c]; break;
    case ES_FIELD_OWNER: out[i] = (double)owner[c]; break;
    case ES_FIELD_FLAGS: out[i] = (double)flags[c]; break;
    case ES_FIELD_FB:
        for (int k = 0; k < 3; k++) out[(long long)k * n + i] = (double)fb[k * N + c];
        break;
    case ES_FIELD_PDF:
    case ES_FIELD_PDF_LAST: {
        const S* f = which == ES_FIELD_PDF ? cur : last;
        for (int q = 0; q < 19; q++) out[(long long)q * n + i] = Store<S>::to_f(q, f[q * ps + c]);
        break;
    }
    case ES_FIELD_RHO:
    case ES_FIELD_U: {
        double r = 0.0, j0 = 0.0, j1 = 0.0, j2 = 0.0;
        for (int q = 0; q < 19; q++) {
            double v = Store<S>::to_f(q, cur[q * ps + c]);
            r += v;
            j0 += cx(q) * v;
            j1 += cy(q) * v;
            j2 += cz(q) * v;
        }
        if (which == ES_FIELD_RHO) {
            out[i] = r;
        } else {
            out[i] = j0 - 0.5 * ((double)fb[c] + ax);
            out[(long long)n + i] = j1 - 0.5 * ((double)fb[N + c] + ay);
            out[2LL * n + i] = j2 - 0.5 * ((double)fb[2 * N + c] + az);
        }
        break;
    }
    }
}

unsigned blocks_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

template <class S>
Streams<S> streams(const es_ctx* c) {
    Streams<S> P;
    const S* src = (const S*)c->pdf[c->cur];
    S* dst = (S*)c->pdf[1 - c->cur];
    for (int q = 0; q < 19; q++) {
        P.src[q] = src + (size_t)q * (size_t)c->g.ps;
        P.dst[q] = dst + (size_t)q * (size_t)c->g.ps;
    }
    return P;
}

// Calls fn with a value of the context's PDF storage type (double, float or
// __half) so that a generic lambda can instantiate the kernel for it.
template <class Fn>
void dispatch_store(const es_ctx* c, Fn&& fn) {
    if (c->P.precision == ES_MIXED16)
        fn(__half{});
    else if (mixed(c))
        fn(0.0f);
    else
        fn(0.0);
}

// The stream-collide's block shape (es_params.lbm_block; 0 = 32 x 4: a warp
// per row segment and four rows a block, so that the rows y +- 1 of psi the
// fused body force reads are mostly in the block's own L1; measured at 512^3
// 3.79 ms against 3.85 for 32 x 2 and 64 x 2, 3.86 for 32 x 8, 4.09 for 128 x
// 2).
dim3 lbm_block(const es_ctx* c) {
    if (c->P.lbm_block[0] <= 0) return dim3(32, 4);
    return dim3(c->P.lbm_block[0], c->P.lbm_block[1] > 0 ? c->P.lbm_block[1] : 1);
}

cudaError_t launch_lbm(es_ctx* c) {
    const Grid& g = c->g;
    const dim3 blk = lbm_block(c);
    const dim3 grd((g.nx + blk.x - 1) / blk.x, (g.ny + blk.y - 1) / blk.y, g.nz);
    const double* a = c->P.accel;
    // the body force evaluated in the stream-collide: first the stored values
    // of the cells next to obstacles and walls
    const bool lazy = c->fb_lazy;
    if (lazy) {
        const cudaError_t e = launch_body_force_near(c);
        if (e != cudaSuccess) return e;
    }
    const double k2e = c->S.kappa * c->S.kappa * c->S.eps;
    const FbPsi fp{c->psi32, (float)c->P.E_ext[0], (float)c->P.E_ext[1], (float)c->P.E_ext[2], (float)k2e};
    dispatch_store(c, [&](auto tag) {
        using S = decltype(tag);
        using C = typename Store<S>::C;
        // algorithmic bytes per cell: 19 populations in and out, f_b (3 C)
        // or psi (4) and the flag byte in
        ProfScope ps(c, "lbm", -1, (double)g.N * (38.0 * sizeof(S) + (lazy ? 4.0 : 3.0 * sizeof(C)) + 1.0));
        const bool per = g.per[0] && g.per[1] && g.per[2];
        auto run = [&](auto slip, auto fused) {
            constexpr bool SL = decltype(slip)::value, FB = decltype(fused)::value;
            auto k = per ? k_lbm<S, false, FB, true> : k_lbm<S, SL, FB, false>;
            launch_pdl(c, k, grd, blk, 0, g, streams<S>(c),
                       (const uint8_t*)c->flags, (const int32_t*)c->owner, (const DParticle*)c->part,
                       (const float*)c->partf, (const C*)c->fb, (C)a[0], (C)a[1], (C)a[2],
                       trt<C>(c->lambda_e, c->lambda_o), c->slip, fp);
        };
        using T_ = std::true_type;
        using F_ = std::false_type;
        if constexpr (std::is_same<C, float>::value) {
            if (lazy) {
                if (c->slip)
                    run(T_{}, T_{});
                else
                    run(F_{}, T_{});
                return;
            }
        }
        if (c->slip)
            run(T_{}, F_{});
        else
            run(F_{}, F_{});
    });
    count(c);
    return cudaGetLastError();
}

// The stream-collide of n contexts (same precision and device, no
// free-slip faces; checked by the caller) in one launch on cs[0]'s stream,
// ordered after each context's pending work and before its later work by
// events.  Each context's per-run preparation (the body force at cells next
// to obstacles) runs on its own stream first.
cudaError_t launch_lbm_batch(es_ctx* const* cs, int n) {
    cudaStream_t bs = cs[0]->stream;
    for (int i = 0; i < n; i++) {
        es_ctx* c = cs[i];
        if (c->fb_lazy) {
            const cudaError_t e = launch_body_force_near(c);
            if (e != cudaSuccess) return e;
        }
        if (!c->ev_sync) {
            const cudaError_t e = cudaEventCreateWithFlags(&c->ev_sync, cudaEventDisableTiming);
            if (e != cudaSuccess) return e;
        }
        if (i > 0) {
            cudaError_t e = cudaEventRecord(c->ev_sync, c->stream);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(bs, c->ev_sync, 0);
            if (e != cudaSuccess) return e;
        }
    }
    cudaError_t err = cudaSuccess;
    dispatch_store(cs[0], [&](auto tag) {
        using S = decltype(tag);
        using C = typename Store<S>::C;
        BatchTable<S> T;
        long long tiles = 0;
        double cells = 0.0;
        for (int i = 0; i < n; i++) {
            es_ctx* c = cs[i];
            BatchRun<S>& R = T.r[i];
            R.g = c->g;
            R.P = streams<S>(c);
            R.flags = c->flags;
            R.owner = c->owner;
            R.part = c->part;
            R.partf = c->partf;
            R.fb = (const C*)c->fb;
            R.ax = (C)c->P.accel[0];
            R.ay = (C)c->P.accel[1];
            R.az = (C)c->P.accel[2];
            R.R = trt<C>(c->lambda_e, c->lambda_o);
            const double k2e = c->S.kappa * c->S.kappa * c->S.eps;
            R.fp = FbPsi{c->psi32, (float)c->P.E_ext[0], (float)c->P.E_ext[1], (float)c->P.E_ext[2], (float)k2e};
            R.lazy = c->fb_lazy ? 1 : 0;
            R.tiles_x = (c->g.nx + kBatchTileX - 1) / kBatchTileX;
            R.tiles_y = (c->g.ny + kBatchTileY - 1) / kBatchTileY;
            R.tile0 = tiles;
            tiles += (long long)R.tiles_x * R.tiles_y * c->g.nz;
            cells += (double)c->g.N;
        }
        T.n = n;
        T.ntiles = tiles;
        const long long cap = (long long)cs[0]->n_sm * 16;
        const unsigned grid = (unsigned)(tiles < cap ? tiles : cap);
        ProfScope ps(cs[0], "lbm_batch", -1, cells * (38.0 * sizeof(S) + 4.0 + 1.0));
        k_lbm_batch<S><<<grid, kBatchTileX * kBatchTileY, 0, bs>>>(T);
        count(cs[0]);
        err = cudaGetLastError();
    });
    if (err != cudaSuccess) return err;
    err = cudaEventRecord(cs[0]->ev_sync, bs);
    for (int i = 1; i < n && err == cudaSuccess; i++) err = cudaStreamWaitEvent(cs[i]->stream, cs[0]->ev_sync, 0);
    return err;
}

template <class S, int T>
cudaError_t run_forces(es_ctx* c, int src, double rmax) {
    const double* E = c->P.E_ext;
    // room for the cells with links of a sphere whose rows fit the bit words
    // (R <= 13.5): their centres lie between R and R + sqrt 2 of its centre, so
    // they number less than the volume between R - 1.9 and R + 2.4
    const double r = rmax < 13.5 ? rmax : 13.5, ro = r + 2.4, ri = r > 1.9 ? r - 1.9 : 0.0;
    const int room = (int)(4.19 * (ro * ro * ro - ri * ri * ri)) + 32;
    // (and for a pass over the fields of a larger one)
    const int least = rmax > 12.0 ? kForceEach * T : kForceChunk;
    const int cells = room < least ? least : (room + 7) / 8 * 8;
    auto launch = [&](auto* kernel, size_t lists, size_t most) -> cudaError_t {
        // (the attribute belongs to the kernel: the most any context needs)
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (e != cudaSuccess) return e;
        launch_pdl(c, kernel, c->np, T, lists, c->g, (const DParticle*)c->part, (const int32_t*)c->owner,
                   (const uint8_t*)c->flags, (const S*)c->pdf[src], E[0], E[1], E[2], (const double*)c->mapped,
                   c->F, c->T, cells);
        return cudaGetLastError();
    };
    const size_t words = (size_t)2 * kForceSide * kForceSide * 4, list = (size_t)cells * 8, most = 12 * 1024 * 8;
    if constexpr (std::is_same<S, double>::value)
        return launch(k_forces<T>, words + list, words + most);
    else
        return launch(k_forces_f32<S, T>, words + list + (size_t)kForceLinks * 8, words + most + kForceLinks * 8);
}

cudaError_t launch_forces(es_ctx* c) {
    if (c->np == 0) return cudaSuccess;
    int src = c->last_src >= 0 ? c->last_src : c->cur;
    ProfScope ps(c, "forces", -1, 0.0);
    double rmax = 0.0;
    for (double r : c->h_R) rmax = r > rmax ? r : rmax;
    cudaError_t err = cudaSuccess;
    dispatch_store(c, [&](auto tag) {
        using S = decltype(tag);
        // few spheres: a block of 1,024 threads each
        err = c->np <= 2 * c->n_sm ? run_forces<S, 1024>(c, src, rmax) : run_forces<S, 256>(c, src, rmax);
    });
    count(c);
    return err;
}

// A new particle state from the host: position, velocities, zeta, q and the
// charge of the Coulomb force (Eq. SurfChrgZetaRelationDebHuck for a zeta
// sphere) replace the record's; the surface charge density found by the last
// mapping stays until the next one recomputes it, and the mass and moment of
// inertia follow from the fixed radius.  In the MIXED32 form the sphere's
// boundary value (2 zeta, or sigma / eps) is split into float-float as the
// mapping does.
__global__ void k_set_particles(const double* __restrict__ in, DParticle* part, const int* kind, double eps,
                                double* pbd, float* pbc, float* __restrict__ pf, int np) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    const double* s = in + 12 * p;
    DParticle& d = part[p];
    for (int a = 0; a < 3; a++) {
        d.x[a] = s[a];
        d.v[a] = s[3 + a];
        d.w[a] = s[6 + a];
    }
    if (pf)
        for (int k = 0; k < 9; k++) pf[12 * p + k] = (float)s[k];
    d.zeta = s[9];
    d.q = s[10];
    d.qeff = s[11];
    const double bv = kind[p] == ES_KIND_ZETA ? 2.0 * d.zeta : d.sigma / eps;
    if (pbd) pbd[p] = bv;
    if (pbc) {
        const ff v = ff_from_double(bv);
        pbc[2 * p] = v.hi;
        pbc[2 * p + 1] = v.lo;
    }
}

cudaError_t launch_set_particles(es_ctx* c) {
    if (c->np == 0) return cudaSuccess;
    k_set_particles<<<blocks_for(c->np, 128), 128, 0, c->stream>>>(c->pstage, c->part, c->kind, c->S.eps, c->pbd, c->pbc,
                                                                   c->partf, c->np);
    count(c);
    return cudaGetLastError();
}

cudaError_t launch_advance(es_ctx* c) {
    if (c->np == 0) return cudaSuccess;
    ProfScope ps(c, "advance", -1, 0.0);
    launch_pdl(c, k_advance, blocks_for(3 * (long long)c->np, 128), 128, 0, c->np, c->part, (const double*)c->F,
               (const double*)c->T, c->g.per[0], c->g.per[1], c->g.per[2], (double)c->g.nx, (double)c->g.ny,
               (double)c->g.nz, c->partf);
    count(c);
    return cudaGetLastError();
}

cudaError_t launch_particles_f32(es_ctx* c) {
    if (!mixed(c) || c->np == 0) return cudaSuccess;
    k_particles_f32<<<(c->np + 127) / 128, 128, 0, c->stream>>>(c->np, c->part, c->partf);
    count(c);
    return cudaGetLastError();
}

cudaError_t launch_fill_rest(es_ctx* c) {
    const int N = (int)c->g.N;
    dim3 grd((N + 255) / 256, 19);
    dispatch_store(c, [&](auto tag) {
        using S = decltype(tag);
        k_fill_rest<S><<<grd, 256, 0, c->stream>>>(N, (size_t)c->g.ps, (S*)c->pdf[0], (S*)c->pdf[1]);
    });
    count(c);
    return cudaGetLastError();
}

cudaError_t launch_get_pdf(es_ctx* c, int buf, double* dst) {
    long long n = 19 * c->g.N;
    dispatch_store(c, [&](auto tag) {
        using S = decltype(tag);
        k_get_pdf<S><<<blocks_for(n, 256), 256, 0, c->stream>>>(c->g.N, c->g.ps, (const S*)c->pdf[buf], dst);
    });
    count(c);
    return cudaGetLastError();
}

cudaError_t launch_set_pdf(es_ctx* c, const double* src) {
    long long n = 19 * c->g.N;
    dispatch_store(c, [&](auto tag) {
        using S = decltype(tag);
        k_set_pdf<S><<<blocks_for(n, 256), 256, 0, c->stream>>>(c->g.N, c->g.ps, src, (S*)c->pdf[c->cur]);
    });
    count(c);
    return cudaGetLastError();
}

cudaError_t launch_get_moments(es_ctx* c, double* rho, double* u) {
    const Grid& g = c->g;
    const double* a = c->P.accel;
    if (!mixed(c)) {
        const double *f = (const double*)c->pdf[c->cur], *fb = (const double*)c->fb;
        if (rho) k_moments<true><<<blocks_for(g.N, 256), 256, 0, c->stream>>>(g.N, g.ps, f, fb, a[0], a[1], a[2], rho);
        if (u) k_moments<false><<<blocks_for(g.N, 256), 256, 0, c->stream>>>(g.N, g.ps, f, fb, a[0], a[1], a[2], u);
        count(c, (rho ? 1 : 0) + (u ? 1 : 0));
        return cudaGetLastError();
    }
    const bool lazy = c->fb_lazy;
    if (u && lazy) {
        const cudaError_t err = launch_body_force_near(c);
        if (err != cudaSuccess) return err;
    }
    const double k2e = c->S.kappa * c->S.kappa * c->S.eps;
    const FbPsi fp{c->psi32, (float)c->P.E_ext[0], (float)c->P.E_ext[1], (float)c->P.E_ext[2], (float)k2e};
    Accel3 acc;
    for (int k = 0; k < 3; k++) acc.a[k] = ff_from_double(-0.5 * a[k]);
    const dim3 blk(32, 8), grd((g.nx + 31) / 32, (g.ny + 7) / 8, g.nz);
    dispatch_store(c, [&](auto tag) {
        using S = decltype(tag);
        if constexpr (!std::is_same<S, double>::value) {
            const S* f = (const S*)c->pdf[c->cur];
            const float* fb = (const float*)c->fb;
            if (rho) k_moments_ff<S, true, false><<<grd, blk, 0, c->stream>>>(g, f, fb, c->flags, fp, acc, rho);
            if (u && lazy)
                k_moments_ff<S, false, true><<<grd, blk, 0, c->stream>>>(g, f, fb, c->flags, fp, acc, u);
            else if (u)
                k_moments_ff<S, false, false><<<grd, blk, 0, c->stream>>>(g, f, fb, c->flags, fp, acc, u);
        }
    });
    count(c, (rho ? 1 : 0) + (u ? 1 : 0));
    return cudaGetLastError();
}

cudaError_t launch_set_fb(es_ctx* c, const double* src) {
    c->fb_lazy = false;  // (the given field is used until the next solve)
    long long n = 3 * c->g.N;
    if (mixed(c))
        k_load_fb<float><<<blocks_for(n, 256), 256, 0, c->stream>>>(n, src, (float*)c->fb);
    else
        k_load_fb<double><<<blocks_for(n, 256), 256, 0, c->stream>>>(n, src, (double*)c->fb);
    count(c);
    return cudaGetLastError();
}

cudaError_t launch_get_fb(es_ctx* c, double* dst) {
    const cudaError_t err = materialize_body_force(c);
    if (err != cudaSuccess) return err;
    long long n = 3 * c->g.N;
    if (mixed(c))
        k_copy_fb<float><<<blocks_for(n, 256), 256, 0, c->stream>>>(n, (const float*)c->fb, dst);
    else
        k_copy_fb<double><<<blocks_for(n, 256), 256, 0, c->stream>>>(n, (const double*)c->fb, dst);
    count(c);
    return cudaGetLastError();
}

cudaError_t launch_gather(es_ctx* c, int which, const long long* idx, int n, double* out) {
    if (which == ES_FIELD_FB || which == ES_FIELD_U) {
        const cudaError_t err = materialize_body_force(c);
        if (err != cudaSuccess) return err;
    }
    const double* a = c->P.accel;
    int last = c->last_src >= 0 ? c->last_src : c->cur;
    dispatch_store(c, [&](auto tag) {
        using S = decltype(tag);
        using C = typename Store<S>::C;
        k_gather<S><<<blocks_for(n, 128), 128, 0, c->stream>>>(
            which, c->g.N, c->g.ps, idx, n, (const S*)c->pdf[c->cur], (const S*)c->pdf[last], (const C*)c->fb,
            c->psi, c->psi32, c->psi_lo, c->owner, c->flags, a[0], a[1], a[2], out);
    });
    count(c);
    return cudaGetLastError();
}

}  // namespace es
