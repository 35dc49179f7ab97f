// The FP64 tile: the phases of stage_tile (stage_kernel.cuh) with
// everything linear on the integer pipe. Primitives and cell fluxes are kept
// in shared memory taken apart (fx::split: 64-bit integer and exponent), so a
// face's stencils are aligned to their own scale by a shift each; face states
// (fixed_face.cuh), flux reconstruction and the viscous gradients are integer
// sums, and so are the primitives and the cell fluxes (fixed_math.cuh). FP64
// arithmetic remains for the Riemann solver, the viscous flux, the stage update
// and the limiter of the few faces beside strong jumps (wide_face.cuh). With CONS
// (MEG7-cons) the planes taken apart are the conservative variables, and the
// primitives of the cells beside faces are kept as they are.
#pragma once

#include "stage_kernel.cuh"
#include "wide_face.cuh"

namespace gbr {

template <int BX, int BY, bool VISC, bool CONS = false, bool TMA = true>
struct FixedLayout {
    using G = TileLayout<BX, BY, VISC>;  // index ranges
    typedef long long i64;
    static constexpr int NU = G::NU, NFX = G::NFX, NFY = G::NFY;
    static constexpr size_t up(size_t b) { return (b + 127) / 128 * 128; }
    static constexpr size_t oM = 0;                                          // reconstructed variables: integers [4][NU]
    static constexpr size_t oFX = oM + sizeof(i64) * 4 * NU;                 // x fluxes [4][NFX]
    static constexpr size_t oFY = oFX + sizeof(i64) * 4 * NFX;               // y fluxes [4][NFY]
    // The FP64 tile + halo lands here; viscous gradients and face fluxes, all
    // written after phase 0, take its place.
    static constexpr size_t oRaw = up(oFY + sizeof(i64) * 4 * NFY);
    static constexpr size_t oGX = oRaw, oGY = oGX + (VISC ? sizeof(double) * 4 * G::NGX : 0);
    static constexpr size_t oHX = oGY + (VISC ? sizeof(double) * 4 * G::NGY : 0);
    static constexpr size_t oHY = oHX + sizeof(double) * 4 * G::NHX;
    static constexpr size_t oH1 = oHY + sizeof(double) * 4 * G::NHY, oR1 = oRaw + (TMA ? sizeof(double) * 4 : sizeof(float)) * NU;
    static constexpr size_t oW = oH1 > oR1 ? oH1 : oR1;                      // CONS: u, v, p of cells [5, B + 7) [3][NW]
    static constexpr int WW = BX + 2, NW = WW * (BY + 2);
    // densities in FP32 [NU], read before the face fluxes are written
    static constexpr size_t oR = TMA || VISC ? oW + (CONS ? sizeof(double) * 3 * NW : 0) : oRaw;
    static constexpr size_t oE = TMA || VISC ? oR + sizeof(float) * NU : oW + (CONS ? sizeof(double) * 3 * NW : 0);  // exponents of the integers above
    static constexpr size_t oEX = oE + sizeof(short) * 4 * NU;
    static constexpr size_t oEY = oEX + sizeof(short) * 4 * NFX;
    static constexpr size_t oPX = oEY + sizeof(short) * 4 * NFY;             // detector flags
    static constexpr size_t oPY = oPX + G::NPX;
    static constexpr size_t bytes = (oPY + G::NPY + 15) / 16 * 16;
};

// Eq. detector's test (trouble_cell) at FP32 cost: the comparison is taken on
// the densities rounded to FP32 wherever the rounding cannot change its sign
// (all but a few cells in a thousand), else on the FP64 values as trouble_cell
// takes it (`exact`). With |r| <= R each density is off by at most 2^-24 R, a
// and b (sums of two differences, three roundings) by at most d = 24 2^-24 R,
// and t = (a^2 + b^2 + eps) - 2 (2ab + eps) by at most 8 d (a + b) + 6 d^2 plus
// the roundings of t itself, below 2^-21 of its terms.
template <typename F>
__device__ __forceinline__ bool trouble_filtered(const float* r, int st, F exact)
{
    const float eps = float(0.9 * 0.5 / (1.0 - 0.9 * 0.5) * 1e-6);
    const float c = r[0], m1 = r[-st], m2 = r[-2 * st], p1 = r[st], p2 = r[2 * st];
    const float a = fabsf(c - m1) + fabsf(fmaf(-2.f, m1, c) + m2);
    const float b = fabsf(c - p1) + fabsf(fmaf(-2.f, p1, c) + p2);
    const float R = fmaxf(fmaxf(fmaxf(fabsf(c), fabsf(m1)), fmaxf(fabsf(m2), fabsf(p1))), fabsf(p2));
    const float d = 24.f / 16777216.f * R, ab = a * b, sq = fmaf(a, a, b * b);
    const float t = (sq + eps) - 2.f * fmaf(2.f, ab, eps);
    const float off = fmaf(8.f * d, a + b, 6.f * d * d) + (sq + 4.f * ab + 3.f * eps) * (1.f / 2097152.f);
    if (t > off) return true;
    if (t < -off) return false;
    return exact();  // (also where a density overflows FP32)
}

// The viscous part of the face flux (viscous_flux, with its terms collected),
// subtracted from out. alpha-damping with alpha_v = 4 takes the normal
// derivative as (2 d - s / 2) / h, d the difference and s the sum of the two
// cells' values and dx-scaled gradients; with s at 60 times its value that is
// (2 / h) (d - s / 240). T = gamma v, v = p / rho, v' = (p' - v rho') / rho. In all
// 29 FP64 operations where the terms one by one take 63 (viscous 1280 x 640 step
// 2.09 -> 1.87 ms), the factors from the host.
template <bool CONS, typename V>
__device__ __forceinline__ void fixed_viscous(const FaceIn<double>& in, const double (&u0)[4], const double (&u1)[4],
                                              double gm1, const V& k, double (&out)[4])
{
    const double ir0 = fx::rcp(u0[0]), ir1 = fx::rcp(u1[0]);
    double dr[2] = {in.g[0][0], in.g[0][in.sg]}, dn[2] = {in.g[1][0], in.g[1][in.sg]};
    double dt[2] = {in.g[2][0], in.g[2][in.sg]}, dp[2] = {in.g[3][0], in.g[3][in.sg]};
    double gn[2] = {in.tun[0], in.tun[in.stq]}, gt[2] = {in.tut[0], in.tut[in.stq]};
    if constexpr (CONS) {  // primitive gradients from the conservative ones (chain rule)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const double n = c ? u1[1] : u0[1], t = c ? u1[2] : u0[2], ir = c ? ir1 : ir0;
            const double k2 = rmul(0.5, rfma(n, n, rmul(t, t)));
            dp[c] = rmul(gm1, rfma(k2, dr[c], rfma(-t, dt[c], rfma(-n, dn[c], dp[c]))));
            dn[c] = rmul(rfma(-n, dr[c], dn[c]), ir);
            dt[c] = rmul(rfma(-t, dr[c], dt[c]), ir);
            const double ra = in.tr0[c ? in.stq : 0];
            gn[c] = rmul(rfma(-n, ra, gn[c]), ir);
            gt[c] = rmul(rfma(-t, ra, gt[c]), ir);
        }
    }
    constexpr double h = -1.0 / 240.0;
    const double v0 = rmul(u0[3], ir0), v1 = rmul(u1[3], ir1);
    const double e0 = rmul(rfma(-v0, dr[0], dp[0]), ir0), e1 = rmul(rfma(-v1, dr[1], dp[1]), ir1);
    const double un = rfma(h, dn[0] + dn[1], u1[1] - u0[1]), ut = rfma(h, dt[0] + dt[1], u1[2] - u0[2]);
    const double tn = rfma(h, e0 + e1, v1 - v0);
    const double tau_nn = rfma(k.nn, un, -rmul(k.ntt, gt[0] + gt[1])), tau_nt = rfma(k.nt, ut, rmul(k.tn, gn[0] + gn[1]));
    out[1] -= tau_nn;
    out[2] -= tau_nt;
    const double w = rfma(tau_nn, u0[1] + u1[1], rmul(tau_nt, u0[2] + u1[2]));
    out[3] = rfma(-k.q, tn, rfma(-0.5, w, out[3]));
}

// The flagged faces of a tile (list: ns whose states, then from L::NF nt whose shear
// velocities are) shared out among all warps, eight a warp: rho, un and p to S,
// ut to T (two planes each).
template <typename L, int BX, int NT, int ORDER>
__device__ __noinline__ void fixed_share(const long long* m, const unsigned short* e, const unsigned short* list, int ns, int nt,
                                         double gamma, double* S, double* T)
{
    const int tid = threadIdx.x, js = (ns + 7) / 8, jobs = js + (nt + 7) / 8;
    for (int job = tid >> 5; job < jobs; job += NT / 32) {
        const bool states = job < js;
        const int at = 8 * (states ? job : job - js) + ((tid & 31) >> 2), n = states ? ns : nt, k = tid & 3;
        const int w = list[(states ? 0 : L::NF) + min(at, n - 1)];
        const bool xf = w < L::NHX, keep = at < n && k < 2;
        const int w2 = xf ? w : w - L::NHX, fw = xf ? L::HXW : BX, fr = w2 / fw, fc = w2 - fr * fw;
        const int c = (fr + (xf ? 6 : 5)) * L::RW + fc + (xf ? 5 : 6);
        const fx::Face f{m + c, e + c, xf ? 1 : L::RW, L::NU, xf ? 1 : 2};
        const fx::WideLanes lanes{(tid & 31) & 28};
        if (states) {
            double r, u, p;
            fx::wide_states<ORDER>(lanes, f, gamma, r, u, p);
            if (keep) {
                S[k * L::NF + w] = r;
                S[(2 + k) * L::NF + w] = u;
                S[(4 + k) * L::NF + w] = p;
            }
        } else {
            const double u = fx::wide_shear<ORDER>(lanes, f);
            if (keep) T[k * L::NF + w] = u;
        }
    }
}

// Whether a CTA has a second thread for every face (whole warps of them).
constexpr bool fixed_splits_faces(int faces, int threads) { return threads >= 2 * ((faces + 31) / 32 * 32); }

template <int BX, int BY, int NT, bool VISC, int ORDER, bool TMA, bool CONS = false, bool MAP = false>
__device__ __forceinline__ void fixed_tile(const StageParams& P, const int tx0, const int ty0, unsigned char* smem,
                                           const CUtensorMap* tmap = nullptr)
{
    typedef long long i64;
    typedef unsigned short u16;
    using F = FixedLayout<BX, BY, VISC, CONS, TMA>;
    using L = typename F::G;
    using X = typename L::template Cross<0>;  // the staged cells
    constexpr int RW = L::RW, NU = L::NU, V = L::V;
    i64* const sM = reinterpret_cast<i64*>(smem + F::oM);
    i64* const sFX = reinterpret_cast<i64*>(smem + F::oFX);
    i64* const sFY = reinterpret_cast<i64*>(smem + F::oFY);
    double* const sGX = reinterpret_cast<double*>(smem + F::oGX);
    double* const sGY = reinterpret_cast<double*>(smem + F::oGY);
    double* const sHX = reinterpret_cast<double*>(smem + F::oHX);
    double* const sHY = reinterpret_cast<double*>(smem + F::oHY);
    double* const sW = reinterpret_cast<double*>(smem + F::oW);
    float* const sR = reinterpret_cast<float*>(smem + F::oR);
    u16* const sE = reinterpret_cast<u16*>(smem + F::oE);
    u16* const sEX = reinterpret_cast<u16*>(smem + F::oEX);
    u16* const sEY = reinterpret_cast<u16*>(smem + F::oEY);
    unsigned char* const sPX = smem + F::oPX;
    unsigned char* const sPY = smem + F::oPY;
    const int nx = P.g.nx, ny = P.g.ny, tid = threadIdx.x;

    PhysT<double> ph;
    ph.gamma = P.ph.gamma;
    ph.gm1 = P.ph.gm1;
    ph.igm1 = P.ph.igm1;
    ph.mu = P.ph.mu;
    ph.kq = P.ph.kq;
    ph.lm = P.ph.riemann;
    const double inv_dx = P.ph.inv_dx, inv_dy = P.ph.inv_dy;
    const fx::Pos gamma = fx::pos(ph.gamma), gm1 = fx::pos(ph.gm1);
    __shared__ double step_dt;
    stage_scalars<MAP>(P, &step_dt);

    // Phase 0: primitives (Eq. pressure) and cell fluxes F^c = (rho u, rho u u
    // + p, rho u v, u (E + p)), G^c (Sec. 1; rho u, rho v, E from the state).
    const bool staged = stage_region<BX, BY, NT, X, TMA, MAP>(
        P, tx0, ty0, reinterpret_cast<double*>(smem + F::oRaw), tmap,
        [&](int idx, double q0, double q1, double q2, double q3) {
            fx::Cell w;
            fx::cell_of(q0, q1, q2, q3, gm1, w);
            const int ry = idx / RW, rx = idx - ry * RW;
            auto put = [&](int m, const fx::Split& x) { fx::store(x, sM[m * NU + idx], sE[m * NU + idx]); };
            put(0, w.r);
            if constexpr (CONS) {
                put(1, w.ru);
                put(2, w.rv);
                put(3, fx::split(q3));
                if (ry >= 5 && ry < BY + 7 && rx >= 5 && rx < BX + 7) {
                    const int c = (ry - 5) * F::WW + rx - 5;
                    sW[c] = fx::unsplit(w.u.m, w.u.e);
                    sW[F::NW + c] = fx::unsplit(w.v.m, w.v.e);
                    sW[2 * F::NW + c] = fx::unsplit(w.p.m, w.p.e);
                }
            } else {
                put(1, w.u);
                put(2, w.v);
                put(3, w.p);
            }
            sR[idx] = f64_to_f32_rn(q0);
            if (ry >= 6 && ry < 6 + BY && rx >= 1 && rx < BX + 11) {
                const int f = (ry - 6) * L::FXW + (rx - 1);
                auto flux = [&](int m, const fx::Split& x) { fx::store(x, sFX[m * L::NFX + f], sEX[m * L::NFX + f]); };
                flux(0, w.ru);
                flux(1, fx::sum(w.ruu, w.p));
                flux(2, fx::product(w.ru, w.v));
                flux(3, fx::product(w.u, w.h));
            }
            if (ry >= 1 && ry < BY + 11 && rx >= 6 && rx < BX + 6) {
                const int f = (ry - 1) * BX + (rx - 6);
                auto flux = [&](int m, const fx::Split& x) { fx::store(x, sFY[m * L::NFY + f], sEY[m * L::NFY + f]); };
                flux(0, w.rv);
                flux(1, fx::product(w.rv, w.u));
                flux(2, fx::sum(w.rvv, w.p));
                flux(3, fx::product(w.v, w.h));
            }
        });
    if (!staged) return;
    __syncthreads();

    constexpr int HALF = NT / 2;
    static_assert(NT % 32 == 0, "whole warps");
    constexpr bool SPLIT = fixed_splits_faces(L::NF, NT);
    __shared__ double sT[SPLIT ? 6 * L::NF : 1];  // ut L, ut R, F of the face
    auto meet = [] { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };  // (reached from both halves' code)
    // There too the faces of wide_face.cuh are shared out among all warps, by lists
    // of those whose states or shear velocities are flagged: one CTA an SM waits for
    // the slowest of its warps (pass of four steps, each warp its own / shared: double
    // Mach 60 x 24 468 / 335 us, viscous 100 x 50 502 / 393, four-quadrant 60 x 60 279
    // / 248, 64^2 vortex, which has none, 45.1 / 45.4 a step; as part of the kernel
    // instead of a call 51.6, the code of a short launch being fetched as it runs).
    constexpr bool SHARE = SPLIT && !CONS;
    __shared__ double sS[SHARE ? 6 * L::NF : 1];  // rho L, R, un L, R, p L, R of a flagged face
    __shared__ u16 sList[SHARE ? 2 * L::NF : 1];
    __shared__ int sCount[2];
    auto share = [&] {  // after both halves have met; true: they meet again
        const int ns = sCount[0], nt = sCount[1];
        if (ns + nt > 0) fixed_share<L, BX, NT, ORDER>(sM, sE, sList, ns, nt, ph.gamma, sS, sT);
        return ns + nt > 0;
    };

    // Phase 1: detector flags, and the gradients the viscous flux takes.
    auto flag = [&](int c, int st) {
        return trouble_filtered(sR + c, st, [&] {
            double r[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) r[k] = fx::unsplit(sM[c + (k - 2) * st], sE[c + (k - 2) * st]);  // (exact: rho is the state's)
            return trouble_cell(r + 2, 1);
        }) ? 1 : 0;
    };
    if (SHARE && tid < 2) sCount[tid] = 0;
    for (int idx = tid; idx < L::NPX; idx += NT) {
        const int a = idx / L::PXW, b = idx - a * L::PXW;
        sPX[idx] = flag((a + 6) * RW + (b + 3), 1);
    }
    for (int idx = tid; idx < L::NPY; idx += NT) {
        const int a = idx / BX, b = idx - a * BX;
        sPY[idx] = flag((a + 3) * RW + (b + 6), RW);
    }
    if constexpr (VISC) {
        auto gradient = [&](int m, int c, int st) {
            i64 q[7];
            int e[7];
#pragma unroll
            for (int k = 0; k < 7; ++k) {
                q[k] = sM[m * NU + c + (k - 3) * st];
                e[k] = sE[m * NU + c + (k - 3) * st];
            }
            return fx::grad60(q, e);
        };
        for (int idx = tid; idx < L::NGX; idx += NT) {
            const int a = idx / L::GXW, b = idx - a * L::GXW;
            for (int m = 0; m < 4; ++m) sGX[m * L::NGX + idx] = gradient(m, (a + 6 - V) * RW + (b + 3), 1);
        }
        for (int idx = tid; idx < L::NGY; idx += NT) {
            const int a = idx / L::GYW, b = idx - a * L::GYW;
            for (int m = 0; m < 4; ++m) sGY[m * L::NGY + idx] = gradient(m, (a + 3) * RW + (b + 6 - V), RW);
        }
    }
    __syncthreads();

    // Phase 2: every x face and y face of the tile, once (one thread per face; in
    // a tile with threads for it, a second one per face, a whole half of the CTA,
    // evaluates what the states do not need, the shear field and the flux
    // reconstruction: where one small tile is all an SM has, a face's chain of
    // dependent instructions is the time, 64^2 step 50.0 -> 44.8 us).
    // Whole warps: a lane past the last face repeats it and stores nothing.
    for (int item = tid; item < (SPLIT ? NT : (L::NF + 31) / 32 * 32); item += NT) {
        const bool second = SPLIT && item >= HALF;
        const int wa = second ? item - HALF : item;
        const bool live = wa < L::NF;
        const int w = live ? wa : L::NF - 1;
        const bool xf = w < L::NHX;
        const int w2 = xf ? w : w - L::NHX;
        const int fw = xf ? L::HXW : BX;
        const int fr = w2 / fw, fc = w2 - fr * fw;                // x faces: row, face; y faces: face, column
        const int c = (fr + (xf ? 6 : 5)) * RW + fc + (xf ? 5 : 6);  // the cell before the face
        const int su = xf ? 1 : RW;
        const int pn = xf ? 1 : 2;  // plane of the normal velocity
        // Eq. buffer: sigma = 0 if psi_k < psi_c for any k in j-2..j+3.
        const unsigned char* tr = xf ? sPX + fr * L::PXW + fc + 2 : sPY + (fr + 2) * BX + fc;
        const int st = xf ? 1 : BX;
        bool trouble = false;
#pragma unroll
        for (int k = -2; k <= 3; ++k) trouble |= tr[k * st] != 0;

        auto plane = [&](int m) { return m == 1 ? pn : m == 2 ? 3 - pn : m; };
        const int cw = (fr + (xf ? 1 : 0)) * F::WW + fc + (xf ? 0 : 1), sw = xf ? 1 : F::WW;
        auto cell = [&](int m, int o) {  // variable m of the cell before (o = 0) or after (su) the face
            if (CONS && m > 0) return sW[(plane(m) - 1) * F::NW + cw + (o ? sw : 0)];
            const int at = plane(m) * NU + c + o;
            return fx::unsplit(sM[at], sE[at]);
        };
        auto value = [&](int m, int o) {
            const int at = plane(m) * NU + c + o;
            fx::Split x;
            x.m = sM[at];
            x.e = sE[at];
            return x;
        };
        auto load = [&](int m, fx::Stencil& x) {
            const int at = plane(m) * NU + c;
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                x.m[k] = sM[at + (k - 5) * su];
                x.e[k] = sE[at + (k - 5) * su];
            }
        };
        const fx::WideFace face{sM, sE, NU, RW, c, xf};  // for the few faces of wide_face.cuh
        auto any = [](bool b) { return __any_sync(0xffffffffu, b); };
        double Fs[4];
        auto reconstruct = [&] {  // the central part where sigma = 1 (Sec. 2.4)
            const int at = xf ? fr * L::FXW + fc + 4 : (fr + 4) * BX + fc, sf = xf ? 1 : BX;
            const int nf = xf ? L::NFX : L::NFY;
            const i64* fm = (xf ? sFX : sFY) + at;
            const u16* fe = (xf ? sEX : sEY) + at;
#pragma unroll 1
            for (int m = 0; m < 4; ++m) {
                const int pl = (m == 1 ? pn : m == 2 ? 3 - pn : m) * nf;
                i64 q[10];
                int e[10];
#pragma unroll
                for (int k = 0; k < 10; ++k) {
                    q[k] = fm[pl + (k - 4) * sf];
                    e[k] = fe[pl + (k - 4) * sf];
                }
                const double f = fx::recon_mean<ORDER>(q, e);
                if (m == 0) Fs[0] = f;
                if (m == 1) Fs[1] = f;
                if (m == 2) Fs[2] = f;
                if (m == 3) Fs[3] = f;
            }
        };
        if constexpr (SPLIT) {
            if (second) {
                double ut[2] = {0.0, 0.0};
                if constexpr (!CONS) {
                    bool wide;
                    const int still = fx::still_exponent(sE[c], sE[3 * NU + c], sE[c + su], sE[3 * NU + c + su]);
                    const bool in_range = fx::shear_states<ORDER>(load, still, ut, wide);
                    if (wide && in_range && live) sList[L::NF + atomicAdd(&sCount[1], 1)] = (u16)w;
                    if (!in_range) ut[0] = __longlong_as_double(0x7ff8000000000000ll);  // refused
                }
                if (!trouble) reconstruct();
                if (live) {
                    sT[w] = ut[0];
                    sT[L::NF + w] = ut[1];
                    if (!trouble) {
#pragma unroll
                        for (int m = 0; m < 4; ++m) sT[(2 + m) * L::NF + w] = Fs[m];
                    }
                }
                meet();
                if constexpr (SHARE) {
                    if (share()) meet();
                }
                break;
            }
        }
        // Characteristic projection at the arithmetic-mean state, every
        // factor from one reciprocal square root y = 1/sqrt(gamma p rho).
        // (Twice the means: X = (2 rho)(2 gamma p), y = 1/sqrt(X) = 1/(2 rho c),
        // 1/c = 2 rho y, 2 rho c = X y.)
        const fx::Split rs = fx::sum(value(0, 0), value(0, su));
        fx::Split ps;
        if constexpr (!CONS) ps = fx::sum(value(3, 0), value(3, su));
        else ps = fx::split(cell(3, 0) + cell(3, su));
        const bool positive = rs.m > 0 && ps.m > 0;  // (else the fallback below)
        const fx::Pos rb = fx::pos(positive ? rs.m : 1, rs.e), gp = gamma * fx::pos(positive ? ps.m : 1, ps.e);
        const fx::Pos xx = gp * rb, y = fx::rsqrt(xx), icb = rb * y, ic2 = icb * icb;
        double rL, unL, utL, pL, rR, unR, utR, pR;
        bool ok;
        if constexpr (!CONS) {
            fx::FaceStates s;
            fx::face_states<ORDER, !SPLIT>(load, y, xx * y, ic2, s);
            const bool wide = s.ok && s.wide && positive;
            if constexpr (SPLIT) {
                if (wide && live) sList[atomicAdd(&sCount[0], 1)] = (u16)w;
                meet();
                if (share()) meet();
                s.ut[0] = sT[w];
                s.ut[1] = sT[L::NF + w];
                s.ok = s.ok && fx::exponent(s.ut[0]) != 2047;
                if (wide) {
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        s.r[k] = sS[k * L::NF + w];
                        s.un[k] = sS[(2 + k) * L::NF + w];
                        s.p[k] = sS[(4 + k) * L::NF + w];
                    }
                }
            } else {
                const bool wide_ut = s.ok && s.wide_ut;
                if (any(wide_ut)) fx::wide_shear_warp<ORDER>(face, wide_ut, s.ut);
                if (any(wide)) fx::wide_states_warp<ORDER>(face, wide, ph.gamma, s);
            }
            rL = s.r[0], unL = s.un[0], utL = s.ut[0], pL = s.p[0];
            rR = s.r[1], unR = s.un[1], utR = s.ut[1], pR = s.p[1];
            ok = s.ok;
        } else {
            const double ub = rmul(0.5, cell(1, 0) + cell(1, su)), vb = rmul(0.5, cell(2, 0) + cell(2, su));
            const double cb = fx::to_double(gp * y), ic = fx::to_double(icb);
            fx::ConsCoefs C;
            C.b1 = fx::to_double(gm1 * ic2);
            C.b1u = rmul(C.b1, ub);
            C.b1v = rmul(C.b1, vb);
            C.b2 = rmul(0.5, rfma(C.b1u, ub, rmul(C.b1v, vb)));
            C.uc = rmul(ub, ic);
            C.ic = ic;
            C.v = vb;
            fx::ConsStates s;
            fx::cons_states<ORDER>(
                load,
                [&](int m) {
                    const int at = plane(m) * NU + c;
                    int e = fx::kExpMin;
#pragma unroll
                    for (int k = -5; k <= 6; ++k) e = max(e, (int)sE[at + k * su]);
                    return e;
                },
                C, s);
            const bool wide_w3 = s.ok && s.wide_w3, wide = s.ok && s.wide && positive;
            if (any(wide_w3)) fx::wide_cons_shear_warp<ORDER>(face, wide_w3, C.v, s.w3);
            if (any(wide)) fx::wide_cons_states_warp<ORDER>(face, wide, C, s);
            if constexpr (SPLIT) meet();
            ok = s.ok;
            // Back with the right eigenvectors, to primitives: rho un = u rho
            // + c d, rho ut = v rho + w3, so un = u + a, ut = v + b with a =
            // c d / rho, b = w3 / rho, and E - rho (un^2 + ut^2) / 2 =
            // c^2 s / (gamma - 1) - (c d a + w3 b) / 2.
            const double c2 = rmul(cb, cb), hg = -0.5 * ph.gm1;
            auto back = [&](int k, double& r, double& un, double& ut, double& p) {
                r = s.r[k];
                const double ir = fx::rcp(r), cd = rmul(cb, s.d[k]), a = rmul(cd, ir), b = rmul(s.w3[k], ir);
                un = ub + a;
                ut = vb + b;
                p = rfma(hg, rfma(cd, a, rmul(s.w3[k], b)), rmul(c2, s.s[k]));
            };
            back(0, rL, unL, utL, pL);
            back(1, rR, unR, utR, pR);
        }
        // positivity fallback: a face state with rho <= 0 or p <= 0 (or from a
        // refused stencil) takes the adjacent cell's state
        ok = ok && positive;
        if (!(ok && tpositive(rL) && tpositive(pL))) {
            rL = cell(0, 0);
            unL = cell(1, 0);
            utL = cell(2, 0);
            pL = cell(3, 0);
        }
        if (!(ok && tpositive(rR) && tpositive(pR))) {
            rR = cell(0, su);
            unR = cell(1, su);
            utR = cell(2, su);
            pR = cell(3, su);
        }
        // Flux reconstruction (Sec. 2.4).
        if (!live) break;  // (the last round)
        if constexpr (SPLIT) {
#pragma unroll
            for (int m = 0; m < 4; ++m) Fs[m] = trouble ? 0.0 : sT[(2 + m) * L::NF + w];
        } else if (!trouble) {
            reconstruct();
        }
        double out[4];
        hllc_flux(ph, !trouble, Fs, rL, unL, utL, pL, rR, unR, utR, pR, out);
        if constexpr (VISC) {
            // Primitives (rho, un, ut, p) of the face's two cells
            double u0[4], u1[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                u0[m] = cell(m, 0);
                u1[m] = cell(m, su);
            }
            FaceIn<double> in;
            // gradients along the face normal at the cell before the face, and
            // the tangential derivatives of un and ut
            const double* gn = xf ? sGX + (fr + V) * L::GXW + fc + 2 : sGY + (fr + 2) * L::GYW + fc + V;
            const double* gt = xf ? sGY + (fr + 3) * L::GYW + fc + V - 1 : sGX + (fr - 1 + V) * L::GXW + fc + 3;
            const int nn = xf ? L::NGX : L::NGY, nt = xf ? L::NGY : L::NGX;
            in.g[0] = gn;
            in.g[1] = gn + pn * nn;
            in.g[2] = gn + (3 - pn) * nn;
            in.g[3] = gn + 3 * nn;
            in.sg = xf ? 1 : L::GYW;
            in.tun = gt + pn * nt;
            in.tut = gt + (3 - pn) * nt;
            in.stq = xf ? 1 : L::GXW;
            in.tr0 = gt;
            fixed_viscous<CONS>(in, u0, u1, ph.gm1, P.visc[xf ? 0 : 1], out);
        }
        if (xf) {
#pragma unroll
            for (int m = 0; m < 4; ++m) sHX[m * L::NHX + w] = out[m];
            if (P.sigx) {
                const int i = ty0 + fr, jf = tx0 + fc;
                if (i < ny && jf <= nx) P.sigx[(long long)i * (nx + 1) + jf] = trouble ? 0 : 1;
            }
        } else {
            sHY[w2] = out[0];
            sHY[L::NHY + w2] = out[2];
            sHY[2 * L::NHY + w2] = out[1];
            sHY[3 * L::NHY + w2] = out[3];
            if (P.sigy) {
                const int j = tx0 + fc, iface = ty0 + fr;
                if (j < nx && iface <= ny) P.sigy[(long long)iface * nx + j] = trouble ? 0 : 1;
            }
        }
    }
    __syncthreads();
    finish_tile<double, BX, BY, NT>(P, step_dt, ph, inv_dx, inv_dy, tx0, ty0, sHX, sHY);
}

// The instances of the smallest tile read ghost cells through the boundary
// rules: on the grids that take it a ghost fill before every stage is a
// quarter of the step (64^2: 57 -> 50 us without), where in the larger tiles the
// code for it costs registers that they need (1024^2 2.0% slower with it).
constexpr bool fixed_maps_ghosts(int bx) { return bx == 8; }

constexpr int kMaxTileRows = 65535;  // of a launch's y extent

// One CTA per tile, two CTAs per SM (viscous MEG7-cons: one, by shared memory).
template <int BX, int BY, int NT, bool VISC, int ORDER, bool CONS>
__global__ void __launch_bounds__(NT, CONS && VISC ? 1 : 2)
    fixed_kernel(const StageParams P, const __grid_constant__ CUtensorMap tmap)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    dependent_start();
    const int ty = blockIdx.z * gridDim.y + blockIdx.y;  // (the rows of tiles in planes of at most kMaxTileRows)
    if (ty * BY >= P.g.ny) return;
    fixed_tile<BX, BY, NT, VISC, ORDER, true, CONS, fixed_maps_ghosts(BX)>(P, blockIdx.x * BX, ty * BY, smem_raw, &tmap);
}

template <int BX, int BY, int NT, bool VISC, int ORDER, bool CONS>
cudaError_t launch_fixed_tiles(const StageParams& p, cudaStream_t s)
{
    using F = FixedLayout<BX, BY, VISC, CONS>;
    static PerDevice<int> configured;  // the shared-memory limit is raised once per device
    auto kern = fixed_kernel<BX, BY, NT, VISC, ORDER, CONS>;
    int ok = 0;
    cudaError_t e = configured.get(&ok, [&](int* v) {
        *v = 1;
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F::bytes);
    });
    if (e != cudaSuccess) return e;
    CUtensorMap map;
    e = encode_state_map(p.g, p.q, F::G::RW, F::G::RH, &map);
    if (e != cudaSuccess) return e;
    const int rows = (p.g.ny + BY - 1) / BY, planes = (rows + kMaxTileRows - 1) / kMaxTileRows;
    dim3 grid((p.g.nx + BX - 1) / BX, planes == 1 ? rows : kMaxTileRows, planes);
    return launch_dependent(kern, grid, NT, F::bytes, s, p, map);
}

// The shape of tile_rule.h on the current device.
inline cudaError_t fixed_tile_shape(const Grid& g, bool cons, bool viscous, TileShape* t)
{
    static PerDevice<int> sm_count;
    int sms = 0;
    cudaError_t e = sm_count.get(&sms, [](int* v) {
        int dev = 0;
        const cudaError_t r = cudaGetDevice(&dev);
        return r != cudaSuccess ? r : cudaDeviceGetAttribute(v, cudaDevAttrMultiProcessorCount, dev);
    });
    if (e != cudaSuccess) return e;
    *t = fixed_tile_rule(g.nx, g.ny, sms, cons, viscous);
    return cudaSuccess;
}

template <bool VISC, int ORDER, bool CONS = false>
cudaError_t launch_fixed(const StageParams& p, cudaStream_t s)
{
    TileShape t;
    const cudaError_t e = fixed_tile_shape(p.g, CONS, VISC, &t);
    if (e != cudaSuccess) return e;
    if (t.bx == 8) return launch_fixed_tiles<8, 4, 192, VISC, ORDER, CONS>(p, s);
    if (t.by == 8) return launch_fixed_tiles<16, 8, 288, VISC, ORDER, CONS>(p, s);
    return launch_fixed_tiles<16, 15, 256, VISC, ORDER, CONS>(p, s);
}

}  // namespace gbr
