// CG with Jacobi in block fixed point (bbs_fixed.cuh): Alg. 1 as cg_system and
// cg_packed_system run it, written for the matrix with Jacobi folded in. With
// x~ = D x, p~ = D p and A~ = A D^-1 (unit diagonal) the method is
//   rho = r . D^-1 r ; t = A~ p~ ; alpha = rho / (p~ . D^-1 t) ; x~ += alpha p~ ;
//   r -= alpha t ; p~ = r + (rho' / rho) p~,
// so r, p~, t and x~ share the residual's scale and only the two inner products
// see the diagonal: as (G r).(G r) and (G p~).(G t) with G = D^-1/2, which halves
// its spread. Below the largest G entry the sums keep 57 bits, so a system whose
// diagonal entries differ by more than 2^24 is left to FP64, and so is one with a
// negative entry (no positive definite matrix) or outside what folded_setup takes.
//
// Run on A as it is (z = D^-1 r a vector of its own) the bound was 2^8, and a
// 3-point recipe batch holds systems beyond it (a corner row's diagonal is a single
// draw): those ran both codes one after the other, 300 systems of n = 32 in 353 us
// where FP64 took 212.
#pragma once

#include "bbs_fixed.cuh"

namespace bbs {
namespace fx {

// 1 / sqrt(a), a > 0: an FP32 value and two Newton steps y += y (1 - x y^2) / 2, as
// rcp. x in [1/4, 1) by an even power of two, y 2^61 ~ 1 / sqrt(x) in (1, 2].
__device__ __forceinline__ Sc inv_sqrt(Sc a) {
    const int odd = (a.e + 62) & 1;
    const long long x = a.m >> odd;  // x 2^62
    const float f = fminf(rsqrtf((float)(int)(x >> 31) * 4.656612873077393e-10f), 1.9999998f);
    long long y = (long long)(int)(f * 1073741824.0f) << 31;
    {
        const long long d = (1ll << 60) - mul62(x, mul62(y, y));  // 2^60 (1 - x y^2), below 2^40
        y += wide((int)(y >> 31), (int)(d >> 10), 0) >> 20;
    }
    {
        const long long d = (1ll << 60) - mul62(x, mul62(y, y));  // below 2^20
        y += wide((int)(y >> 31), (int)d, 0) >> 30;
    }
    y = min(max(y, 1ll << 61), (1ll << 62) - 1);
    return Sc{y, -(a.e + 62 + odd) / 2 - 61};
}

// As bicgstab_fixed.
template <int FMT, int SF, int R, class G>
__device__ __forceinline__ Fit cg_fixed(const Mat<double>& A, const Mat<double>& S, const SysIO& io, bool valid, const SolveCfg& C,
                                        const TeamSmem& sm, G g, const Team& team) {
    const int n = io.n;
    Team tm = team;
    if (G::kLanes != 0) tm.nt = G::kLanes;  // (known to the compiler)
    const int2* as = in_shared<int2>(S.vals);
    int2* pa = in_shared<int2>(sm.xa);  // p~
    int2* pb = in_shared<int2>(sm.xb);  // x~ for true residuals
    const bool last = tm.row(R - 1) < n;  // only a lane's last row may lie past the end

    long long X[R], Rv[R];  // x~, r
    int eX, bX, eR, bR, sigma;
    bool run;
    Sc nb2;
    if (!folded_setup<FMT, SF, kCg>(A, S, io, valid, sm, g, tm, X, eX, bX, Rv, eR, bR, sigma, run, nb2)) {
        // (the block's other warps count on this one at their barriers)
        for (int it = 1; it <= C.max_iters && g.live(false); ++it) {
        }
        return kUnfit;
    }
    Dig w[R];  // G in units of 2^(eW - 58)
    int eW;
    {
        g.sync();  // pa and pb are spent
        long long* wm = in_shared<long long>(sm.xb);
        int most = -100000;
#pragma unroll 1
        for (int row = tm.tid; row < n; row += tm.nt) {
            const Sc q = inv_sqrt(unpack(diag_entry<FMT>(A, row)));
            wm[row] = q.m;
            pa[row].x = q.e;
            most = max(most, q.e);
        }
        most = g.max_int(most);
        eW = most + 62;
#pragma unroll
        for (int q = 0; q < R; ++q)
            w[q] = q + 1 < R || last ? split(round_shr(wm[tm.row(q)], most + 4 - pa[tm.row(q)].x)) : Dig{0, 0};
    }
    const Sc tol2 = unpack(C.tol * C.tol), tau2 = C.tol_type == 1 ? mul(tol2, nb2) : tol2;
    Sc rr = norm2_full(Rv, eR, g);
    bR = 57;
    // G y, at y's exponent plus eW
    const auto weighted = [&](Dig c, Dig y) -> Dig {
        Sum s{0, 1 << 28};
        s.add(c, y);
        return split(s.value());
    };
    int eP = kNone, bP = 0;
    unsigned op = 0;  // the high digits of the caller's rows of p~, or-ed
    // p~ = r (56 bits) where `take` says so, and r . D^-1 r
    const auto start = [&](bool take) -> Sc {
        Dot d;
        d.clear();
        if (take) op = 0;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const Dig f = split(Rv[q]);
            d.square(weighted(w[q], f));
            if (take && (q + 1 < R || last)) {
                op |= mag(f.hi);
                pa[tm.row(q)] = pack(f);
            }
        }
        const Part pt[1] = {part(d)};
        const int pe[1] = {2 * (eR + eW)};
        Sc r[1];
        unsigned none = 0;
        g.sums(pt, pe, r, none);
        if (take) eP = eR;
        return r[0];
    };
    int status = -1, iters = 0, restarts = 0;
    Sc res2 = rr;
    bool active = run;
    if (active && le(rr, tau2)) {
        status = ST_CONVERGED;
        active = false;
    }
    Sc rho = start(true);

    for (int it = 1; it <= C.max_iters; ++it) {
        if (!g.live(active)) break;
        if (!g.any(active)) continue;
        if (active) {
            iters = it;
            if (!finite(rho)) {
                status = ST_NAN;
                active = false;
            } else if (zero(rho)) {
                status = ST_BREAKDOWN;
                active = false;
            }
        }
        g.sync();
        Dig t[R];
        spmv_fixed<SF, R>(S, as, pa, t, tm);
        const int eT = eP + sigma - 2;
        Sc ptp;
        int bT;
        {
            Dot d;
            d.clear();
            unsigned ot = 0;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const Dig p = q + 1 < R || last ? dig(pa[tm.row(q)]) : Dig{0, 0};
                d.add(weighted(w[q], t[q]), weighted(w[q], p));
                ot |= mag(t[q].hi);
            }
            const Part pt[1] = {part(d)};
            const int pe[1] = {eP + eT + 2 * eW};
            Sc r[1];
            unsigned o = masks(op, ot);
            g.sums(pt, pe, r, o);
            ptp = r[0];
            bP = bits_first(o);
            bT = bits_second(o);
        }
        if (active) {
            if (!finite(ptp)) {
                status = ST_NAN;
                active = false;
            } else if (zero(ptp)) {
                status = ST_BREAKDOWN;
                active = false;
            }
        }
        const Sc alpha = mul(rho, rcp(ptp));
        {  // x~ += alpha p~, kept to 61 bits (a system that has stopped keeps its x~)
            const int eo = max(eX + max(0, bX - 60), eP + ex(alpha) - 2);
            Dig c = coef(alpha, eP, eo);
            if (!active) c = Dig{0, 0};
            shr_rows(X, active ? eo - eX : 0, g);
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) {
                    Sum s{X[q], 1 << 28};
                    s.add(c, dig(pa[tm.row(q)]));
                    X[q] = s.value();
                }
            if (active) eX = eo;
        }
        Sc rho_hat;
        {  // r -= alpha t
            const int eo = max(eR + max(0, bR - 56), eT + ex(alpha) + max(-2, bT - 56));
            const Dig c = coef(neg(alpha), eT, eo);
            shr_rows(Rv, eo - eR, g);
            eR = eo;
            Dot dr, dz;
            dr.clear();
            dz.clear();
            unsigned orr = 0, ox = 0;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                Sum s{Rv[q], 1 << 28};
                s.add(c, t[q]);
                Rv[q] = s.value();
                const Dig f = split(Rv[q]);
                dr.square(f);
                dz.square(weighted(w[q], f));
                orr |= mag(f.hi);
                ox |= mag((int)(X[q] >> 32));
            }
            const Part pt[2] = {part(dr), part(dz)};
            const int pe[2] = {2 * eR, 2 * (eR + eW)};
            Sc r[2];
            unsigned o = masks(orr, ox);
            g.sums(pt, pe, r, o);
            rr = r[0];
            rho_hat = r[1];
            bR = bits_first(o);
            bX = bits_second(o) + 3;  // (of the upper words)
        }
        bool cand = false;
        if (active) {
            if (!finite(rr)) {
                status = ST_NAN;
                active = false;
            } else {
                cand = le(rr, tau2);
            }
        }
        fill_up(Rv, eR, bR, g);
        {  // p~ = r + (rho^ / rho) p~
            const Sc beta = mul(rho_hat, rcp(rho));
            const int eo = max(eR + max(0, bR - 56), eP + ex(beta) + max(-2, bP - 56));
            const Dig c = coef(beta, eP, eo);
            long long y[R];
#pragma unroll
            for (int q = 0; q < R; ++q) y[q] = Rv[q];
            shr_rows(y, eo - eR, g);
            op = 0;
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) {
                    Sum s{y[q], 1 << 28};
                    s.add(c, dig(pa[tm.row(q)]));
                    const Dig f = split(s.value());
                    pa[tm.row(q)] = pack(f);
                    op |= mag(f.hi);
                }
            eP = eo;
        }
        bool restarted = false;
        if (g.any(cand)) {
            const Sc res = true_residual<SF>(S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, cand, g, tm);
            bool again = false;
            if (cand) {
                res2 = res;
                if (!finite(res)) {
                    status = ST_NAN;
                    active = false;
                } else if (le(res, tau2)) {
                    status = ST_CONVERGED;
                    active = false;
                } else if (++restarts > kMaxRestarts) {
                    status = kStagnated;
                    active = false;
                } else {
                    again = true;
                }
            }
            if (g.any(again)) {
                const Sc r0 = start(again);
                if (again) {
                    rho = r0;
                    restarted = true;
                }
            }
        }
        if (!restarted) rho = rho_hat;
    }
    if (active) status = ST_MAX_ITER;
    return folded_finish<FMT, SF>(A, S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, run && accepted(status), iters, status,
                                  status == ST_CONVERGED, res2, tau2, nb2, sm, g, tm)
               ? kDone
               : run ? kLeft : kUnfit;
}

}  // namespace fx

// CG of a block's system: block fixed point where the values are staged, with
// Jacobi, and the system fits it; FP64 otherwise.
template <int FMT, int R>
__global__ void __launch_bounds__(max_threads_for(R), 1) cg_kernel(const SolveParams P) {
    extern __shared__ __align__(16) unsigned char raw[];
    const Team tm = Team::block();
    const int sys = blockIdx.x;
    const auto op = make_op<FMT, R>(P, sys, raw, tm);
    const TeamSmem sm = team_smem(raw, P.n_pad);
    if (op.as != nullptr && P.precond == 1 && tm.nwarps <= fx::kMaxWarps) {
        const Mat<double> S{op.as, op.A.row_ptrs, op.A.cols, op.A.n, op.A.k};
        const fx::Warps g{tm, reinterpret_cast<unsigned char*>(sm.red), 0};
        const fx::Fit fit = fx::cg_fixed<FMT, FMT, R>(op.A, S, sys_io(P, sys), true, solve_cfg(P, sys), sm, g, tm);
        if (fit == fx::kDone) return;
        tm.sync();
        if (fit == fx::kLeft) make_op<FMT, R>(P, sys, raw, tm);
    }
    cg_system<FMT, R>(op, sys_io(P, sys), solve_cfg(P, sys), sm, tm);
}

}  // namespace bbs
