// Per-particle arithmetic of the two gather passes of one right-hand side
// (section 2): the accumulators of particle i, the contribution of one
// neighbour j, the final per-particle formulas, and the loops over a range
// of list entries.  The single-instance and batched pass kernels
// (pair_passes.cu) share them, so an instance's pairs are evaluated with the
// same operations in the same order however it is launched.
#pragma once

#include "debug_checks.cuh"
#include "kernels.cuh"
#include "pair_passes.cuh"
#include "team.cuh"

namespace sph {

// List entries whose neighbour records a mixed-path pass loads together (the
// next ones' indices are on their way meanwhile).  One lane a particle:
// measured at 4.2M on the 1:250 strip, pass A 2, 3, 4 entries 0.99, 0.92,
// 0.93 ms, pass B (its records still two accesses) 1, 2, 3 entries 1.42,
// 0.93, 1.04 ms.  Teams have few iterations: 26k particles, pass A 2, 3
// entries 16.5, 19.8 us, pass B 1, 2 entries 19.0, 20.4 us.
template <int T>
constexpr int UNROLL_A = T == 1 ? 3 : 2;
template <int T>
constexpr int UNROLL_B = T == 1 ? 2 : 1;

// Membership test of a list entry when the lists carry a skin: the exact
// predicate of N(i) on the separation the pass already has (FP32 band test
// with the FP64 predicate inside the band on the mixed path, which alone
// reads i's FP64 values; the FP64 predicate on the FP64 path).
template <typename R, class Args>
__device__ __forceinline__ bool skin_member(const Args &a, R r2, R hi, R hj, int i, int j) {
    if constexpr (sizeof(R) == 4) {
        const float R1 = 3.0f * fmaxf(hi, hj);
        const float R2 = R1 * R1;
        const float band = (R2 + 4.0f * fmaxf(a.an.A[0], a.an.A[1]) * R1) *
                           (1.0f / 65536.0f);
        if (r2 < R2 - band) return true;
        if (r2 > R2 + band) return false;
    }
    return pred_fp64(a.d, __ldg(&a.x[i]), __ldg(&a.y[i]), __ldg(&a.h[i]), __ldg(&a.x[j]),
                     __ldg(&a.y[j]), __ldg(&a.h[j]));
}

// ---------------------------------------------------------------- pass A --
// Summation density (Eq. sd-gather), beta (Eq. beta), p_avg (Eq. pavg, N_i
// counts i), shift dr (Eq. shift-deltar, volume m_j / rho0, W ratio
// against the kernel at its inflection point for h_ij = (h_i + h_j)/2),
// limited to 0.25 h_i (Eq. shift-limit).  finish() also writes the two
// per-particle records pass B gathers: {m, V = m/rho, rho, 1/(rho^2 beta)}
// and {u, v, p, 1/h}.
template <typename R, bool LEAN>
struct PassALane {
    static constexpr bool L64 = lean64<R, LEAN>;
    R hi, hinv, inv_wxi;
    R rho, srw, psum, ax, ay;
    int cnt;

    __device__ __forceinline__ void init(const PassAArgs<R> &a, int i) {
        hi = (R)a.h[i];
        hinv = R(1) / hi;
        inv_wxi = R(1) / qs_w<R>(R(XI_INFLECTION));
        rho = srw = psum = ax = ay = R(0);
        cnt = 0;
    }

    // member j (self: j == i) at separation r_i - r_j = (dx, dy), r2 = r^2
    __device__ __forceinline__ void pair(R mj, R hj, R pj, bool self, R dx,
                                         R dy, R r2) {
        if constexpr (L64) {
            // r = 0 (i itself): rinv = 0 and the shift term is zero
            const R rinv = is_normal(r2) ? frsqrt_lean(r2) : R(0);
            const R r = __dmul_rn(r2, rinv);
            R w, s;
            qs_ws(__dmul_rn(r, hinv), w, s);
            rho += mj * w;
            srw += __dmul_rn(mj, r) * s;  // times -5 in finish()
            psum += pj;
            cnt += 1;
            const R hsinv = frcp(hi + hj);
            qs_ws(__dmul_rn(r + r, hsinv), w, s);
            R ratio = __dmul_rn(w, inv_wxi);
            ratio = __dmul_rn(ratio, ratio);
            // sigma (2 / (h_i + h_j))^3 times -5 s: the constants -40
            // sigma are applied in finish()
            const R f = mj * __fma_rn(__dmul_rn(R(0.24), ratio), ratio, R(1)) *
                        (hsinv * hsinv * hsinv) * __dmul_rn(s, rinv);
            ax += f * dx;
            ay += f * dy;
            return;
        }
        const R rinv = r2 > R(0) ? frsqrt(r2) : R(0);
        const R r = r2 * rinv;
        const R q = r * hinv;
        rho += mj * qs_w<R>(q);
        srw += mj * r * qs_dw<R>(q);
        psum += pj;
        cnt += 1;
        if (!self && r > R(0)) {
            const R hbinv = fdiv(R(2), hi + hj);
            const R qb = r * hbinv;
            R ratio = qs_w<R>(qb) * inv_wxi;
            ratio *= ratio;
            const R f = mj * (R(1) + R(0.24) * ratio * ratio) *
                        (sigma_norm<R>() * hbinv * hbinv * hbinv) *
                        qs_dw<R>(qb) * rinv;
            ax += f * dx;
            ay += f * dy;
        }
    }

    // mixed, LEAN: every kernel term of an entry that is no member (in
    // false) is zero by its clip; constants are applied in finish()
    __device__ __forceinline__ void pair2(R mj, R hj, R pj, bool in, F2 d, R r2,
                                          F2 &acc) {
        const R rinv = frsqrt(fmaxf(r2, F32_LEAST));
        const R r = r2 * rinv;
        const R hsinv = frcp_ftz(hi + hj);
        F2 w, s;
        Qs2(r, f2(-hinv, R(-2) * hsinv)).ws(w, s);
        rho = fmaf(mj, lo(w), rho);
        srw = fmaf(mj * r, lo(s), srw);
        psum += in ? pj : R(0);
        cnt += in ? 1 : 0;
        R ratio = sph::hi(w) * inv_wxi;
        ratio *= ratio;
        const R f = mj * fmaf(R(0.24) * ratio, ratio, R(1)) *
                    (hsinv * hsinv * hsinv) * (sph::hi(s) * rinv);
        acc = fma2(f2(f), d, acc);
    }

    // wall neighbours of particle i (section 2.2): mass m_w in rho, beta
    // and the shift, p_w in p_avg
    template <int T>
    __device__ __forceinline__ void walls(const PassAArgs<R> &a, int i,
                                          const Team<T> &tm) {
        if (a.w.n <= 0) return;
        for_each_wall<T>(a.w, i, a.d, a.an, a.pk[i], a.x[i], a.y[i], a.h[i],
                         tm.lane, tm.mask,
                         [&](int k, double dxd, double dyd, double r2d) {
            pair((R)a.w.m[k], (R)a.w.h[k], (R)a.w.p[k], false, (R)dxd,
                 (R)dyd, (R)r2d);
        });
    }

    template <int T>
    __device__ __forceinline__ void finish(const PassAArgs<R> &a, int i,
                                           const Team<T> &tm) {
        rho = team_sum<T>(tm.mask, rho);
        srw = team_sum<T>(tm.mask, srw);
        psum = team_sum<T>(tm.mask, psum);
        ax = team_sum<T>(tm.mask, ax);
        ay = team_sum<T>(tm.mask, ay);
        cnt = team_sum<T>(tm.mask, cnt);
        if (tm.lane != 0) return;
        // mixed: sigma / h^2 cancels in beta
        [[maybe_unused]] const R beta_lean = R(2.5) * (hinv * srw) / rho;
        if constexpr (LEAN) {
            srw *= R(-5);
            ax *= R(-40) * sigma_norm<R>();
            ay *= R(-40) * sigma_norm<R>();
        }
        const R sig = sigma_norm<R>() * hinv * hinv;
        rho *= sig;
        const R beta = LEAN && !L64 ? beta_lean : -(sig * hinv * srw) / (rho * R(2));
        R drx = R(0), dry = R(0);
        if (beta != R(0)) {
            const R c = R(-0.5) * hi * hi / (R)a.rho0;
            drx = c * ax;
            dry = c * ay;
        }
        R mag;
        if constexpr (L64)
            mag = sqrt(mad2(drx, drx, dry, dry));
        else
            mag = sqrt(drx * drx + dry * dry);
        const R lim = R(0.25) * hi;
        if (mag > lim) {
            const R th = lim / mag;
            drx *= th;
            dry *= th;
        }
        const R mi = a.m[i];
        const R V = mi / rho;
        const R rb2 = beta != R(0) ? R(1) / (rho * rho * beta) : R(0);
        a.rho[i] = rho;
        a.beta[i] = beta;
        a.pavg[i] = psum / (R)cnt;
        a.nnb[i] = cnt;
        a.drx[i] = drx;
        a.dry[i] = dry;
        a.V[i] = V;
        a.rb2[i] = rb2;
        typename V4<R>::T A, B;
        A.x = mi; A.y = V; A.z = rho; A.w = rb2;
        B.x = a.u[i]; B.y = a.v[i]; B.z = a.p[i]; B.w = hinv;
        if constexpr (sizeof(R) == 4) {
            store8(a.nbA + 2 * (size_t)i, A, B);
        } else {
            a.nbA[i] = A;
            a.nbB[i] = B;
        }
    }
};

// ---------------------------------------------------------------- pass B --
// EDAC pressure rate (Eq. edac:sph) and momentum rate (Eq. mom-sph without
// the A_i/A_j stresses and third line, unused per the paper's remark):
//   dp/dt = rho0 c^2/beta_i sum V_j u_ij.gW_i
//         + 1/beta_i sum V_j nu_ij (p_i - p_j) r_ij.gW_ij / (r^2 + eta)
//         + rho_i sum m_j (dr_i/dt).(P_i gW_i + P_j gW_j)
//   du/dt = -sum m_j (P_i gW_i + P_j gW_j)
//         + 1/beta_i sum m_j 4 nu/(rho_i + rho_j) r_ij.gW_ij/(r^2 + eta) u_ij
// gW_i = grad W(r_ij, h_i), gW_ij the mean of gW_i and gW_j (Eq. dw-avg),
// nu_ij the Cleary mean 4 nu_i nu_j/(nu_i + nu_j) of nu_e = alpha_e c h / 8
// (Eqs. edac-alpha, nu-cleary), which equals (alpha_e c / 2) / (1/h_i +
// 1/h_j); eta = 0.001 h_i^2, P_j = (p_j - p_avg,i) / (rho_j^2 beta_j).
// Wall neighbours (section 2.2): prescribed wall velocity in the divergence
// sum, extrapolated velocity in the viscous sum, rho_w = rho0, beta_w = 1.
// Every term carries grad W(r, h_i) or grad W(r, h_j), so a pair with
// r >= 3 max(h_i, h_j) -- or r = 0, i itself -- adds exactly zero.
// Factors common to all pairs of i are applied once, in finish(): the
// Cleary numerator alpha_e c / 2 of the diffusion sum, the 4 nu of the
// viscous sum, and the transport sum, which is (dr_i/dt) . sum m_j (P_i
// gW_i + P_j gW_j) = -(dr_i/dt) . (pressure force sum).
template <typename R, bool LEAN>
struct PassBLane {
    static constexpr bool L64 = lean64<R, LEAN>;
    R hinv, dsig_i, rho_i, pi, ui, vi, pavg_i, Pi, eta;
    bool dden_on, visc_on;
    R div, diff, fax, fay, vx, vy;

    // false: beta_i = 0 (no neighbour at r > 0), zero rates (reading R1)
    __device__ __forceinline__ bool init(const PassBArgs<R> &a, int i) {
        const R rb2i = a.rb2[i];
        const R beta_i = a.beta[i];
        div = diff = fax = fay = vx = vy = R(0);
        if (beta_i == R(0)) return false;
        typename V4<R>::T Bi;
        if constexpr (sizeof(R) == 4)
            Bi = a.nbA[2 * (size_t)i + 1];
        else
            Bi = a.nbB[i];
        hinv = Bi.w;
        dsig_i = L64 ? hinv * hinv * hinv : sigma_norm<R>() * hinv * hinv * hinv;
        rho_i = a.rho[i];
        ui = Bi.x;
        vi = Bi.y;
        pi = Bi.z;
        pavg_i = a.pavg[i];
        Pi = (pi - pavg_i) * rb2i;
        const R hi = R(1) / hinv;
        eta = R(0.001) * hi * hi;
        dden_on = a.diff_denominator != 0;
        visc_on = a.nu != 0.0;
        return true;
    }

    __device__ __forceinline__ static R recip(R b) {
        if constexpr (L64)
            return frcp(b);
        else
            return fdiv(R(1), b);
    }

    // one neighbour's contributions; (ujx, ujy): velocity in the divergence
    // sum, (ugx, ugy): velocity in the viscous sum
    __device__ __forceinline__ void pair(R dx, R dy, R r2, R hjinv, R mj,
                                         R Vj, R rho_j, R Pj, R pj, R ujx,
                                         R ujy, R ugx, R ugy) {
        R gi = 0, gj = 0;
        if constexpr (L64) {
            const R rinv = is_normal(r2) ? frsqrt_lean(r2) : R(0);
            const R r = __dmul_rn(r2, rinv);
            const R k = R(-5) * sigma_norm<R>() * rinv;
            // dsig_i: 1 / h_i^3
            gi = __dmul_rn(qs_s(__dmul_rn(r, hinv)) * k, dsig_i);
            gj = __dmul_rn(qs_s(__dmul_rn(r, hjinv)) * k, hjinv * hjinv * hjinv);
        } else if (r2 > R(0)) {
            const R rinv = frsqrt(r2);
            const R r = r2 * rinv;
            gi = dsig_i * qs_dw<R>(r * hinv) * rinv;
            gj = sigma_norm<R>() * hjinv * hjinv * hjinv *
                 qs_dw<R>(r * hjinv) * rinv;
        }
        const R rdg = R(0.5) * (gi + gj) * r2;
        // nu_ij / (alpha_e c / 2)
        const R nu_ij = recip(hinv + hjinv);
        const R inv_reta = recip(r2 + eta);
        const R uij = ui - ujx, vij = vi - ujy;
        if constexpr (L64)
            div += Vj * gi * mad2(uij, dx, vij, dy);
        else
            div += Vj * gi * (uij * dx + vij * dy);
        diff += Vj * nu_ij * (pi - pj) * rdg * (dden_on ? inv_reta : R(1));
        R mfp;
        if constexpr (L64)
            mfp = mj * mad2(Pi, gi, Pj, gj);
        else
            mfp = mj * (Pi * gi + Pj * gj);
        fax -= mfp * dx;
        fay -= mfp * dy;
        // m_j 4 nu/(rho_i + rho_j) r.gW_ij/(r^2 + eta) / (4 nu)
        // (an inviscid flow's sum is multiplied by zero in finish())
        R visc;
        if constexpr (L64) {
            if (!visc_on) return;
            visc = mj * rdg * inv_reta * frcp(rho_i + rho_j);
        } else {
            visc = fdiv(mj * rdg * inv_reta, rho_i + rho_j);
        }
        vx += visc * (ui - ugx);
        vy += visc * (vi - ugy);
    }

    // mixed, LEAN: the same sums less constant factors, which finish()
    // applies (-5 sigma of both gradients, 1/2 of their mean, the force's
    // sign); sums = {div, diff}, force and viscous vectors
    struct Sums2 {
        F2 f, w;
    };
    __device__ __forceinline__ void pair2(F2 d, const float4 &A, const float4 &B, R pref,
                                          F2 uvi, R hi3, Sums2 &S) {
        const R r2 = fmaf(lo(d), lo(d), hi(d) * hi(d));
        const R rinv = frsqrt(fmaxf(r2, F32_LEAST));
        const F2 g = mul2(mul2(Qs2(r2 * rinv, f2(-hinv, -B.w)).s(), f2(rinv)),
                          f2(hi3, B.w * B.w * B.w));
        const R gi = lo(g), gj = hi(g);
        const R inv_reta = frcp_ftz(r2 + eta);
        const R rdg = (gi + gj) * r2;
        const R rdge = rdg * inv_reta;
        const F2 uv = sub2(uvi, f2(B.x, B.y));
        const F2 ud = mul2(uv, d);
        div = fmaf(A.y * gi, lo(ud) + hi(ud), div);
        diff = fmaf(A.y * frcp_ftz(hinv + B.w) * (dden_on ? rdge : rdg), pi - B.z, diff);
        const R mfp = A.x * fmaf(Pi, gi, (B.z - pref) * A.w * gj);
        S.f = fma2(f2(mfp), d, S.f);
        S.w = fma2(f2(A.x * rdge * frcp_ftz(rho_i + A.z)), uv, S.w);
    }
    __device__ __forceinline__ void take(const Sums2 &S) {
        const R k = R(-5) * sigma_norm<R>();
        div *= k;
        diff *= R(0.5) * k;
        fax = -k * lo(S.f);
        fay = -k * hi(S.f);
        vx = R(0.5) * k * lo(S.w);
        vy = R(0.5) * k * hi(S.w);
    }

    // list neighbour j with its pass-B records A = {m, V, rho, 1/(rho^2
    // beta)}, B = {u, v, p, 1/h}; pref: p_avg,i, or p_avg,j (literal
    // reading, pavg_mode 1)
    template <typename V>
    __device__ __forceinline__ void pair_rec(R dx, R dy, R r2, const V &A,
                                             const V &B, R pref) {
        pair(dx, dy, r2, B.w, A.x, A.y, A.z, (B.z - pref) * A.w, B.z, B.x,
             B.y, B.x, B.y);
    }

    template <int T>
    __device__ __forceinline__ void walls(const PassBArgs<R> &a, int i,
                                          const Team<T> &tm) {
        if (a.w.n <= 0) return;
        const R rho0 = (R)a.rho0;
        const bool literal = a.pavg_mode != 0;
        for_each_wall<T>(a.w, i, a.d, a.an, a.pk[i], a.x[i], a.y[i], a.h[i],
                         tm.lane, tm.mask,
                         [&](int k, double dxd, double dyd, double r2d) {
            const R mk = (R)a.w.m[k], pk = (R)a.w.p[k];
            const R pref = literal ? R(0) : pavg_i;
            pair((R)dxd, (R)dyd, (R)r2d, R(1) / (R)a.w.h[k], mk, mk / rho0,
                 rho0, (pk - pref) / (rho0 * rho0), pk, (R)a.w.uw[k],
                 (R)a.w.vw[k], (R)a.w.ugx[k], (R)a.w.ugy[k]);
        });
    }

    // on: init() returned true (else the rates are zero)
    template <int T>
    __device__ __forceinline__ void finish(const PassBArgs<R> &a, int i,
                                           const Team<T> &tm, bool on) {
        div = team_sum<T>(tm.mask, div);
        diff = team_sum<T>(tm.mask, diff);
        fax = team_sum<T>(tm.mask, fax);
        fay = team_sum<T>(tm.mask, fay);
        vx = team_sum<T>(tm.mask, vx);
        vy = team_sum<T>(tm.mask, vy);
        if (tm.lane != 0) return;
        if (!on) {
            a.dpdt[i] = R(0);
            a.dudt[i] = R(0);
            a.dvdt[i] = R(0);
            return;
        }
        const R beta_i = a.beta[i];
        const R rf = a.rho_factor ? rho_i : R(1);
        // (u~ - u) = dr / dt by the reciprocal the time-step kernel stores
        const R idt = (R)a.dt[1];
        R tvf;
        if constexpr (L64)
            tvf = -mad2(a.drx[i] * idt, fax, a.dry[i] * idt, fay);
        else
            tvf = -(a.drx[i] * idt * fax + a.dry[i] * idt * fay);
        const R half_ac = R(0.5) * (R)a.alpha_e * (R)a.cs;
        const R four_nu = R(4) * (R)a.nu;
        const R dpdt = ((R)a.rho0 * (R)a.cs * (R)a.cs / beta_i) * div +
                       half_ac * diff / beta_i + rf * tvf;
        const R dudt = fax + four_nu * vx / beta_i;
        const R dvdt = fay + four_nu * vy / beta_i;
        a.dpdt[i] = dpdt;
        a.dudt[i] = dudt;
        a.dvdt[i] = dvdt;
        if (!isfinite((double)dpdt) || !isfinite((double)dudt) ||
            !isfinite((double)dvdt))
            atomicOr(a.nonfinite, 1);
    }
};

// The entries of particle i: its row, if the lists have rows, and its list
// behind it, as one sequence (a particle next to a finer level has few row
// entries and many list entries: two loops would each take the warp's
// longest, a third more instructions on the 1:250 strip).
struct Entries {
    const uint32_t *row, *list;   // list: entry k at list[k]
    uint32_t nr, cnt;
    template <class Args>
    __device__ __forceinline__ Entries(const Args &a, int i) {
        nr = a.rows ? __ldg(&a.rlen[i]) & 0xffffu : 0u;
        row = a.rows + ((size_t)(i >> 5) * (32 * a.roww) + (i & 31));
        const uint32_t b = __ldg(&a.off[i]);
        cnt = __ldg(&a.off[i + 1]) - b + nr;
        list = a.list + ((ptrdiff_t)b - (ptrdiff_t)nr);
    }
    __device__ __forceinline__ int at(uint32_t k, int i) const {
        const uint32_t *p = k < nr ? row : list;
        return k < cnt ? (int)__ldg(&p[k < nr ? 32 * k : k]) : i;
    }
};

// Pass A over the entries of particle i, in order (team lane t takes entries
// t, t + T, ...).
template <typename R, int T, bool LEAN>
__device__ __forceinline__ void pass_a_list(const PassAArgs<R> &a, int i,
                                            PassALane<R, LEAN> &L, const Team<T> &tm) {
    Sep<R> sp;
    sp.init(a.d, a.x, a.y, a.pk, i);
    const R hi = L.hi;
    if constexpr (sizeof(R) == 4) {
        // U list entries per step, their records loaded before any is used
        // (more loads in flight per warp)
        [[maybe_unused]] const Sep2 sp2(a.an, sp.pi);
        [[maybe_unused]] F2 acc = f2(0.0f);
        auto body = [&](int j, const float4 &pj, R mj, R pjv) {
            if constexpr (LEAN) {
                // r = 0 (i itself): the gradient sums add zero by s = 0, d = 0
                const F2 d = sp2.get(pj);
                const R r2 = fmaf(lo(d), lo(d), sph::hi(d) * sph::hi(d));
                const bool in = !a.filter || skin_member<R>(a, r2, hi, pj.z, i, j);
                L.pair2(mj, pj.z, pjv, in, d, r2, acc);
                return;
            }
            R dx, dy;
            anchor_sep(a.an, sp.pi, pj, dx, dy);
            const R r2 = fmaf(dx, dx, dy * dy);
            if (a.filter && !skin_member<R>(a, r2, hi, pj.z, i, j))
                return;
            L.pair(mj, pj.z, pjv, j == i, dx, dy, r2);
        };
        constexpr int U = UNROLL_A<T>;
        const Entries E(a, i);
        uint32_t k = tm.lane;
        int jn[U];   // the next entries, loaded ahead of their records
#pragma unroll
        for (int u = 0; u < U; ++u) jn[u] = E.at(k + u * T, i);
        for (; k + (U - 1) * T < E.cnt; k += U * T) {
            int jj[U];
            float4 pp[U];
            R mm[U], qq[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                jj[u] = jn[u];
                // an index out of range (debug builds) reads i instead
                if (!SPH_DCHECK((unsigned)jj[u] < (unsigned)a.n)) jj[u] = i;
                pp[u] = __ldg(&a.pk[jj[u]]);
                mm[u] = a.m[jj[u]];
                qq[u] = a.p[jj[u]];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) jn[u] = E.at(k + (U + u) * T, i);
#pragma unroll
            for (int u = 0; u < U; ++u) body(jj[u], pp[u], mm[u], qq[u]);
        }
#pragma unroll
        for (int u = 0; u < U - 1; ++u) {
            if (k + u * T >= E.cnt) break;
            if (!SPH_DCHECK((unsigned)jn[u] < (unsigned)a.n)) jn[u] = i;
            body(jn[u], __ldg(&a.pk[jn[u]]), a.m[jn[u]], a.p[jn[u]]);
        }
        if constexpr (LEAN) {
            L.ax = lo(acc);
            L.ay = sph::hi(acc);
        }
    } else {
        const Entries E(a, i);   // FP64 steps take exact lists: no rows
        for (uint32_t k = tm.lane; k < E.cnt; k += T) {
            const int j = (int)__ldg(&E.list[k]);
            if (!SPH_DCHECK((unsigned)j < (unsigned)a.n)) continue;
            R dx, dy, r2, hj;
            sp.get(a.d, a.an, a.x, a.y, a.h, a.pk, j, dx, dy, r2, hj);
            if (a.filter && !skin_member<R>(a, r2, hi, hj, i, j))
                continue;
            L.pair(a.m[j], hj, a.p[j], j == i, dx, dy, r2);
        }
    }
}

// Pass B over the entries of particle i, in order.
template <typename R, int T, bool LEAN>
__device__ __forceinline__ void pass_b_list(const PassBArgs<R> &a, int i,
                                            PassBLane<R, LEAN> &L, const Team<T> &tm) {
    Sep<R> sp;
    sp.init(a.d, a.x, a.y, a.pk, i);
    const R pavg_i = L.pavg_i;
    const bool literal = a.pavg_mode != 0;
    const R hpk = (R)a.pk[i].z;   // h_i as the list builder saw it
    if constexpr (sizeof(R) == 4) {
        // neither a membership test for skin entries nor a test for i
        // itself: both add exactly zero
        [[maybe_unused]] const Sep2 sp2(a.an, sp.pi);
        [[maybe_unused]] const F2 uvi = f2(L.ui, L.vi);
        [[maybe_unused]] const R hi3 = L.hinv * L.hinv * L.hinv;
        [[maybe_unused]] typename PassBLane<R, LEAN>::Sums2 S{f2(0.0f), f2(0.0f)};
        auto body = [&](int j, const float4 &pj, const float4 &A,
                        const float4 &B) {
            if constexpr (LEAN) {
                L.pair2(sp2.get(pj), A, B, literal ? a.pavg[j] : pavg_i, uvi, hi3, S);
                return;
            }
            R dx, dy;
            anchor_sep(a.an, sp.pi, pj, dx, dy);
            L.pair_rec(dx, dy, fmaf(dx, dx, dy * dy), A, B,
                       literal ? a.pavg[j] : pavg_i);
        };
        constexpr int U = UNROLL_B<T>;
        const Entries E(a, i);
        uint32_t k = tm.lane;
        int jn[U];   // the next entries, loaded ahead of their records
#pragma unroll
        for (int u = 0; u < U; ++u) jn[u] = E.at(k + u * T, i);
        for (; k + (U - 1) * T < E.cnt; k += U * T) {
            int jj[U];
            float4 pp[U], AA[U], BB[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                jj[u] = jn[u];
                // an index out of range (debug builds) reads i instead
                if (!SPH_DCHECK((unsigned)jj[u] < (unsigned)a.n)) jj[u] = i;
                pp[u] = __ldg(&a.pk[jj[u]]);
                load8(a.nbA + 2 * (size_t)jj[u], AA[u], BB[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) jn[u] = E.at(k + (U + u) * T, i);
#pragma unroll
            for (int u = 0; u < U; ++u) body(jj[u], pp[u], AA[u], BB[u]);
        }
#pragma unroll
        for (int u = 0; u < U - 1; ++u) {
            if (k + u * T >= E.cnt) break;
            if (!SPH_DCHECK((unsigned)jn[u] < (unsigned)a.n)) jn[u] = i;
            float4 A, B;
            load8(a.nbA + 2 * (size_t)jn[u], A, B);
            body(jn[u], __ldg(&a.pk[jn[u]]), A, B);
        }
        if constexpr (LEAN) L.take(S);
    } else {
        const Entries E(a, i);   // FP64 steps take exact lists: no rows
        for (uint32_t k = tm.lane; k < E.cnt; k += T) {
            const int j = (int)__ldg(&E.list[k]);
            if (!SPH_DCHECK((unsigned)j < (unsigned)a.n)) continue;
            if (j == i) continue;
            R dx, dy, r2;
            if (a.filter) {
                R hj;
                sp.get(a.d, a.an, a.x, a.y, a.h, a.pk, j, dx, dy, r2, hj);
                if (!skin_member<R>(a, r2, hpk, hj, i, j))
                    continue;
            } else {
                sp.get(a.d, a.an, a.x, a.y, a.pk, j, dx, dy, r2);
            }
            L.pair_rec(dx, dy, r2, a.nbA[j], a.nbB[j], literal ? a.pavg[j] : pavg_i);
        }
    }
}

}  // namespace sph
