// CG with Jacobi in block fixed point (bbs_fixed.cuh): Alg. 1 as cg_system and
// cg_packed_system run it, on the matrix as it is (no folding: a symmetric
// matrix stays one) and z = D^-1 r formed from the inverse diagonal's digits.
//
// The matrix has one scale, 2^(60 - sigma) with row sums below 2^sigma, so a row
// keeps 60 bits less what its entries lie below the largest row sum; a system
// whose smallest diagonal entry is more than 2^8 below it is left to FP64 (52
// bits at least, FP64's own). Same for systems with a zero or missing diagonal
// entry, non-finite entries, numbers beyond FP32's range or a right-hand side or
// guess beyond 2^+-400.
#pragma once

#include "bbs_fixed.cuh"

namespace bbs {
namespace fx {

// As bicgstab_fixed.
template <int SF, int R, class G>
__device__ __forceinline__ Fit cg_fixed(const Mat<double>& A, const Mat<double>& S, const SysIO& io, bool valid, const SolveCfg& C,
                                         const TeamSmem& sm, G g, const Team& team) {
    const int n = io.n;
    Team tm = team;
    if (G::kLanes != 0) tm.nt = G::kLanes;  // (known to the compiler)
    int2* as = in_shared<int2>(S.vals);
    int2* pa = in_shared<int2>(sm.xa);  // p
    int2* pb = in_shared<int2>(sm.xb);  // x for true residuals
    const bool last = tm.row(R - 1) < n;  // only a lane's last row may lie past the end

    // --- does the system fit?
    long long X[R], Rv[R];
    int eX = kNone, bX = 0, eR, bR, sigma, eD;
    bool run;
    Sc nb2;
    Dig di[R];  // D^-1 in units of 2^(eD - 58), below 4
    {
        long long* dm = in_shared<long long>(sm.xb);  // 1 / a_ii
        int2* de = pa;
        int bad = 0, eb = 0, exm = 0, top = 0, inv = 0;
#pragma unroll 1
        for (int row = tm.tid; row < n; row += tm.nt) {
            double d = 0.0;
            float t = 0.0f;
            each_entry<SF>(S, row, [&](int e, int col) {
                const double v = S.vals[e];
                if (col == row) d = v;
                if (col >= 0) t += fabsf((float)v);
            });
            bad |= normal64(d) ? 0 : 1;
            const Sc q = rcp(unpack(d));
            dm[row] = q.m;
            de[row] = make_int2(q.e, 0);
            inv = max(inv, __float_as_int(fabsf(__frcp_rn((float)d))) & 0x7fffffff);
            top = max(top, __float_as_int(t * 1.0001f) & 0x7fffffff);
            eb = max(eb, (__double2hiint(io.b[row]) >> 20) & 0x7ff);
            const double x0 = io.x[row];
            exm = max(exm, zero64(x0) ? 0 : max(1, (__double2hiint(x0) >> 20) & 0x7ff));
        }
        top = g.max_int(bad ? 0x7fffffff : top);
        inv = g.max_int(inv);
        eb = g.max_int(eb);
        exm = g.max_int(exm);
        const bool xz = exm == 0;  // the guess is zero
        // (row sums within 2^+-100, the largest at most 2^8 times the smallest diagonal)
        run = valid && top > 0x0d800000 && top < 0x71800000 &&
              __int_as_float(top) * __int_as_float(inv) < 256.0f && eb > 623 && eb < 1423 &&
              (xz || (exm > 623 && exm < 1423));
        if (!g.any(run)) {  // (the block's other warps count on this one at their barriers)
            for (int it = 1; it <= C.max_iters && g.live(false); ++it) {
            }
            return kUnfit;
        }
        sigma = (top >> 23) - 126;  // row sums < 2^sigma
        eD = (inv >> 23) - 126 - 1;  // |1 / a_ii| < 2^(eD + 1)
        const int ebq = eb - 1022 - 57;
#pragma unroll
        for (int q = 0; q < R; ++q)
            di[q] = q + 1 < R || last ? split(round_shr(dm[tm.row(q)], eD - 58 - de[tm.row(q)].x)) : Dig{0, 0};
        g.sync();  // dense digits by columns overwrite values that other lanes have read
#pragma unroll 1
        for (int row = run ? tm.tid : n; row < n; row += tm.nt) {
            if (SF == FMT_DENSE && by_columns(n)) {
#pragma unroll 2
                for (int j = 0; j < n; ++j)
                    as[j * n + row] = pack(split(to_int(ldg(A.vals + (size_t)row * n + j), 60 - sigma)));
            } else {
                each_entry<SF>(S, row, [&](int e, int col) {
                    as[e] = pack(split(col >= 0 ? to_int(S.vals[e], 60 - sigma) : 0));
                });
            }
        }
        g.sync();
        eR = ebq;
        bR = 57;
        Dot d;
        d.clear();
#pragma unroll
        for (int q = 0; q < R; ++q) {
            Rv[q] = q + 1 < R || last ? to_int(io.b[tm.row(q)], -ebq) : 0;
            X[q] = 0;
            d.square(split(Rv[q]));
        }
        const Part pt[1] = {part(d)};
        const int pe[1] = {2 * ebq};
        Sc r[1];
        unsigned none = 0;
        g.sums(pt, pe, r, none);
        nb2 = r[0];
        if (g.any(run && !xz)) {
            if (!xz) {
                eX = exm - 1022 - 57;
                bX = 57;
#pragma unroll
                for (int q = 0; q < R; ++q)
                    if (q + 1 < R || last) X[q] = to_int(io.x[tm.row(q)], -eX);
            }
            true_residual<SF>(S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, !xz, g, tm);
        }
    }
    const Sc tol2 = unpack(C.tol * C.tol), tau2 = C.tol_type == 1 ? mul(tol2, nb2) : tol2;
    Sc rr = norm2_full(Rv, eR, g);
    bR = 57;
    // r.z with z = D^-1 r (z at exponent eR + eD, below 2^58), and p = z / 2 where
    // `take` says so
    int eP = kNone, bP = 0;
    unsigned op = 0;  // the high digits of the caller's rows of p, or-ed
    const auto preconditioned = [&](bool take) -> Sc {
        Dot d;
        d.clear();
        if (take) op = 0;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const Dig f = split(Rv[q]);
            Sum s{0, 1 << 28};
            s.add(di[q], f);
            const Dig z = split(s.value());
            d.add(f, z);
            if (take && (q + 1 < R || last)) {
                const Dig h = split((s.value() + 1) >> 1);
                op |= mag(h.hi);
                pa[tm.row(q)] = pack(h);
            }
        }
        const Part pt[1] = {part(d)};
        const int pe[1] = {2 * eR + eD};
        Sc r[1];
        unsigned none = 0;
        g.sums(pt, pe, r, none);
        if (take) eP = eR + eD + 1;
        return r[0];
    };
    int status = -1, iters = 0, restarts = 0;
    Sc res2 = rr;
    bool have_res = true, active = run;
    if (active) {
        if (le(rr, tau2)) {
            status = ST_CONVERGED;
            active = false;
        } else {
            have_res = false;
        }
    }
    Sc rho = preconditioned(true);

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
                d.add(t[q], q + 1 < R || last ? dig(pa[tm.row(q)]) : Dig{0, 0});
                ot |= mag(t[q].hi);
            }
            const Part pt[1] = {part(d)};
            const int pe[1] = {eP + eT};
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
        {  // x += alpha p, kept to 61 bits (a system that has stopped keeps its x)
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
        Dig z[R];
        int eZ, bZ;
        {  // r to 56 bits, r -= alpha t, z = D^-1 r
            fill_up(Rv, eR, bR, g);
            const int eo = max(eR + max(0, bR - 56), eT + ex(alpha) + max(-2, bT - 56));
            const Dig c = coef(neg(alpha), eT, eo);
            shr_rows(Rv, eo - eR, g);
            eR = eo;
            eZ = eR + eD;
            Dot dr, dz;
            dr.clear();
            dz.clear();
            unsigned orr = 0, oz = 0, ox = 0;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                Sum s{Rv[q], 1 << 28};
                s.add(c, t[q]);
                Rv[q] = s.value();
                const Dig f = split(Rv[q]);
                Sum u{0, 1 << 28};
                u.add(di[q], f);
                z[q] = split(u.value());
                dr.square(f);
                dz.add(f, z[q]);
                orr |= mag(f.hi);
                oz |= mag(z[q].hi);
                ox |= mag((int)(X[q] >> 32));
            }
            const Part pt[2] = {part(dr), part(dz)};
            const int pe[2] = {2 * eR, eR + eZ};
            Sc r[2];
            unsigned long long o = (unsigned long long)masks(oz, 0) << 32 | masks(orr, ox);
            g.sums(pt, pe, r, o);
            rr = r[0];
            rho_hat = r[1];
            bR = bits_first((unsigned)o);
            bX = bits_second((unsigned)o) + 3;  // (of the upper words)
            bZ = bits_first((unsigned)(o >> 32));
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
        {  // p = z + (rho^ / rho) p, to 56 bits: z is shifted up where it holds fewer (an
           // inverse diagonal below its largest entry's size), or p, A p and r would
           // lose these bits again every iteration
            const Sc beta = mul(rho_hat, rcp(rho));
            const int eo = max(max(eZ + bZ - 56, eZ - 31), eP + ex(beta) + max(-2, bP - 56));
            const int kz = max(0, eZ - eo);
            const Dig c = coef(beta, eP, eo);
            long long w[R];
#pragma unroll
            for (int q = 0; q < R; ++q) w[q] = shl31(join(z[q]), kz);
            shr_rows(w, max(0, eo - eZ), g);
            op = 0;
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) {
                    Sum s{w[q], 1 << 28};
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
                have_res = true;
                if (!finite(res2)) {
                    status = ST_NAN;
                    active = false;
                } else if (le(res2, tau2)) {
                    status = ST_CONVERGED;
                    active = false;
                } else if (++restarts > kMaxRestarts) {
                    status = kStagnated;
                    active = false;
                } else {
                    have_res = false;
                    again = true;
                }
            }
            if (g.any(again)) {
                const Sc r0 = preconditioned(again);
                if (again) {
                    rho = r0;
                    restarted = true;
                }
            }
        }
        if (!restarted) rho = rho_hat;
    }
    if (active) status = ST_MAX_ITER;
    const bool done = run && accepted(status), need = done && !have_res;
    if (g.any(need)) {
        const Sc res = true_residual<SF>(S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, false, g, tm);
        if (need) res2 = res;
    }
    const bool moved = done && iters > 0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int row = tm.row(q);
        if (moved && row < n) {
            const double x = to_double(normal(X[q], eX));
            io.x[row] = x;
            const Sc xr = unpack(x);
            X[q] = round_shr(xr.m, eX - xr.e);
        }
    }
    // where that rounding weighs in the residual, the log takes the rounded x's
    const bool close = moved && le(res2, Sc{nb2.m, nb2.e - 76});
    if (g.any(close)) {
        const Sc res = true_residual<SF>(S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, false, g, tm);
        if (close) res2 = res;
    }
    if (done && tm.tid == 0) {
        *io.iters = iters;
        *io.rel_res = sqrt(to_double(res2) / to_double(nb2));
        *io.status = status;
        if (io.inner != nullptr) *io.inner = 0;
    }
    return done ? kDone : run ? kLeft : kUnfit;
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
        const fx::Fit fit = fx::cg_fixed<FMT, R>(op.A, S, sys_io(P, sys), true, solve_cfg(P, sys), sm, g, tm);
        if (fit == fx::kDone) return;
        tm.sync();
        if (fit == fx::kLeft) make_op<FMT, R>(P, sys, raw, tm);
    }
    cg_system<FMT, R>(op, sys_io(P, sys), solve_cfg(P, sys), sm, tm);
}

}  // namespace bbs
