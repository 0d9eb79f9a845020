// GMRES(m) with Jacobi folded into the staged matrix in block fixed point
// (bbs_fixed.cuh), for packed systems: the method and the tests of
// gmres_packed_system. The basis vectors have unit norm, so they are digits at
// exponent -57, in the workspace where the FP64 form keeps its basis; the
// orthogonalisation (an inner product and an update for each basis vector) and
// the products with the matrix are integer multiply-adds. The Hessenberg, the
// rotations and the norms' roots stay FP64, on the group's first lane.
//
// 16,384 systems of n = 144 (5-point, CSR, 16 lanes, m = 10): 5.51 ms in FP64,
// 2.79 ms. Bound by latency: the projections' reductions follow one another, and
// so do the first lane's FP64 rotations.
#pragma once

#include "bbs_fixed.cuh"

namespace bbs {
namespace fx {

// As bicgstab_fixed. ext: the group's
// small arrays, as gmres_packed_system lays them out.
template <int FMT, int SF, int R, class G>
__device__ __forceinline__ Fit gmres_fixed(const Mat<double>& A, const Mat<double>& S, const SysIO& io, bool valid,
                                            const SolveCfg& C, const TeamSmem& sm, double* ext_generic, G g,
                                            const Team& team) {
    const int n = io.n, m = C.restart;
    Team tm = team;
    if (G::kLanes != 0) tm.nt = G::kLanes;  // (known to the compiler)
    const int2* as = in_shared<int2>(S.vals);
    int2* pa = in_shared<int2>(sm.xa);  // the basis vector being multiplied
    int2* pb = in_shared<int2>(sm.xb);  // x~ for true residuals
    double* ext = in_shared<double>(ext_generic);
    long long X[R], Rv[R];
    int eX, bX, eR, bR, sigma;
    bool run;
    Sc nb2;
    if (!folded_setup<FMT, SF, kGmres>(A, S, io, valid, sm, g, tm, X, eX, bX, Rv, eR, bR, sigma, run, nb2)) return kUnfit;
    const bool last = tm.row(R - 1) < n;  // only a lane's last row may lie past the end
    // exponent of w = A v and what is left of it: every ||w|| is at most the
    // matrix's Frobenius norm (below 2^fexp), and orthogonalising only shortens w, so
    // that its entries stay below 2^60; nor below the rows' own bound
    int ew0;
    {
        float f2 = 0.0f;
#pragma unroll 1
        for (int row = tm.tid; row < n; row += tm.nt)
            each_entry<SF>(S, row, [&](int e, int) {
                const float h = (float)as[e].x * __int_as_float((127 + 29 - 60 + sigma) << 23);
                f2 = fmaf(h, h, f2);
            });
        const Part pt[1] = {part(Dot{(long long)(f2 * 65600.0f) + 1024, 0, 0})};  // 2^-16 units, rounded up
        const int pe[1] = {-58 - 16};
        Sc r[1];
        unsigned none = 0;
        g.sums(pt, pe, r, none);
        const int fexp = (ex(r[0]) + 1) >> 1;
        ew0 = -57 + max(sigma - 2, fexp - 3);
    }
    const Sc tol2 = unpack(C.tol * C.tol), tau2 = C.tol_type == 1 ? mul(tol2, nb2) : tol2;
    const double tau = sqrt(to_double(tau2));
    Sc beta2 = norm2_full(Rv, eR, g);

    const size_t vs = (size_t)((n + 1) & ~1);
    int2* V = reinterpret_cast<int2*>(C.ws);
    // H column by column, rows 0..j + 1 of column j
    double* H = ext;
    const auto hx = [](int i, int j) { return j * (j + 3) / 2 + i; };
    double* cs = H + m * (m + 3) / 2;
    double* sn = cs + m;
    double* gv = sn + m;
    double* y = gv + m + 1;
    int* ctl = reinterpret_cast<int*>(y + m);
    const bool lead = tm.tid == 0;

    bool active = run;
    int status = -1, it = 0, restarts = 0;
    if (active) {
        if (!finite(beta2)) {
            status = ST_NAN;
            active = false;
        } else if (le(beta2, tau2)) {
            status = ST_CONVERGED;
            active = false;
        }
    }
    while (g.any(active)) {
        if (active && it >= C.max_iters) {
            status = ST_MAX_ITER;
            active = false;
        }
        bool cyc = active;
        const double beta = sqrt(to_double(beta2));
        {  // v_0 = r / beta (r holds 56 bits, so 2 r / beta 2^56 stays below 4)
            const Dig c = coef(unpack(1.0 / beta), eR - 1, -57);
#pragma unroll
            for (int q = 0; q < R; ++q) {
                Sum s{0, 1 << 28};
                s.add(c, split(Rv[q] + Rv[q]));
                if (cyc && (q + 1 < R || last)) V[tm.row(q)] = pack(split(s.value()));
            }
        }
        if (cyc && lead) {
            for (int i = 0; i <= m; ++i) gv[i] = 0.0;
            gv[0] = beta;
        }
        int k = 0;
        bool singular = false, estimate_ok = false;
        for (int j = 0; j < m; ++j) {
            if (!g.any(cyc)) break;
            if (cyc) ++it;
            g.sync();  // every lane is done reading pa
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (q + 1 < R || last) pa[tm.row(q)] = V[(size_t)j * vs + tm.row(q)];
            g.sync();
            long long w[R];
            int ew = ew0;
            {
                Sum s[R];
                spmv_sums<SF, 64>(S, as, pa, s, 1 << 28, tm);
#pragma unroll
                for (int q = 0; q < R; ++q) w[q] = s[q].hh;
                shr_rows(w, ew0 + 59 - sigma, g);
            }
#pragma unroll 1
            for (int i = 0; i <= j; ++i) {  // modified Gram-Schmidt
                Dig vr[R];
                Dot d;
                d.clear();
#pragma unroll
                for (int q = 0; q < R; ++q)
                    vr[q] = q + 1 < R || last ? dig(V[(size_t)i * vs + tm.row(q)]) : Dig{0, 0};
#pragma unroll
                for (int q = 0; q < R; ++q) d.add(split(w[q]), vr[q]);
                const Part pt[1] = {part(d)};
                const int pe[1] = {ew - 57};
                Sc h[1];
                unsigned none = 0;
                g.sums(pt, pe, h, none);
                // (h close to the Frobenius norm)
                const int far = max(0, ex(h[0]) - 59 - ew);
                if (g.any(far > 0)) {
                    shr_rows(w, far, g);
                    ew += far;
                }
                const Dig c = coef(neg(h[0]), -57, ew);
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    Sum s{w[q], 1 << 28};
                    s.add(c, vr[q]);
                    w[q] = s.value();
                }
                if (cyc && lead) H[hx(i, j)] = to_double(h[0]);
            }
            Sc hw[1];
            {
                Dig f[R];
#pragma unroll
                for (int q = 0; q < R; ++q) f[q] = split(w[q]);
                long long carry;
                const Dot d = dot_wide(f, carry);
                const Part pt[1] = {part(d, carry)};
                const int pe[1] = {2 * ew};
                unsigned none = 0;
                g.sums(pt, pe, hw, none);
            }
            // h_{j+1,j} = ||w|| and its reciprocal from one rsqrt
            const double hwd = to_double(hw[0]);
            const double hinv = rsqrt(hwd);
            const double hn = __double_as_longlong(hwd) > 0 ? hwd * hinv : hwd;
            if (cyc && !finite64(hn)) {
                status = ST_NAN;
                active = false;
                cyc = false;
            }
            if (cyc && lead) {
                H[hx(j + 1, j)] = hn;
                for (int i = 0; i < j; ++i) {
                    const double a = H[hx(i, j)], c = H[hx(i + 1, j)];
                    H[hx(i, j)] = cs[i] * a + sn[i] * c;
                    H[hx(i + 1, j)] = -sn[i] * a + cs[i] * c;
                }
                const double a = H[hx(j, j)];
                const double denom = sqrt(a * a + hn * hn);
                int c0, c1 = 0, c2 = 0;
                if (denom == 0.0) {
                    c0 = j;
                    c1 = 1;
                } else {
                    const double dinv = 1.0 / denom;
                    cs[j] = a * dinv;
                    sn[j] = hn * dinv;
                    H[hx(j, j)] = denom;
                    H[hx(j + 1, j)] = 0.0;
                    gv[j + 1] = -sn[j] * gv[j];
                    gv[j] = cs[j] * gv[j];
                    c0 = j + 1;
                    c2 = (hn == 0.0 || fabs(gv[j + 1]) <= tau) ? 1 : 0;
                }
                ctl[0] = c0;
                ctl[1] = c1 | (c2 << 1);
            }
            g.sync();
            if (cyc) {  // the group's first lane wrote its ctl
                k = ctl[0];
                singular = ctl[1] & 1;
                estimate_ok = (ctl[1] >> 1) & 1;
            }
            g.sync();  // ctl is rewritten in the next step
            if (cyc && (singular || estimate_ok || it >= C.max_iters)) cyc = false;
            {  // v_{j+1} = w / ||w||: w shifted up to a norm of 57 bits
                const int up = min(31, max(0, 57 - (((ex(hw[0]) + 1) >> 1) - ew)));
                const Dig c = coef(unpack(hinv), ew - up, -57);
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    Sum s{0, 1 << 28};
                    s.add(c, split(shl31(w[q], up)));
                    if (cyc && (q + 1 < R || last)) V[(size_t)(j + 1) * vs + tm.row(q)] = pack(split(s.value()));
                }
            }
        }
        // y = H(0:k,0:k)^-1 g(0:k) ; x~ += V y, for the groups still solving
        const bool upd = active;
        if (upd && lead) {
            for (int i = k - 1; i >= 0; --i) {
                double sum = gv[i];
                for (int l = i + 1; l < k; ++l) sum -= H[hx(i, l)] * y[l];
                y[i] = sum / H[hx(i, i)];
            }
        }
        g.sync();
        {
            // terms below 2^(ey - eo) each: k of them below 2^60
            const int terms = upd ? k : 0;
            int ey = kNone;
            for (int i = 0; i < terms; ++i) ey = max(ey, ex(unpack(y[i])));
            const int eo = max(eX + max(0, bX - 59), ey - 54);
            shr_rows(X, terms > 0 ? eo - eX : 0, g);
            if (terms > 0) eX = eo;
#pragma unroll 1
            for (int i = 0; g.any(i < terms); ++i) {
                const Dig c = i < terms ? coef(unpack(y[i]), -57, eX) : Dig{0, 0};
#pragma unroll
                for (int q = 0; q < R; ++q)
                    if (i < terms && (q + 1 < R || last)) {
                        Sum s{X[q], 1 << 28};
                        s.add(c, dig(V[(size_t)i * vs + tm.row(q)]));
                        X[q] = s.value();
                    }
            }
            unsigned long long o = 0;
#pragma unroll
            for (int q = 0; q < R; ++q) o |= (unsigned long long)(X[q] ^ (X[q] >> 63));
            bX = g.max_int(64 - __clzll((long long)o));
        }
        if (g.any(upd)) {
            g.sync();
            const Sc res = true_residual<SF>(S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, upd, g, tm);
            if (upd) {
                beta2 = res;
                if (!finite(beta2)) {
                    status = ST_NAN;
                    active = false;
                } else if (le(beta2, tau2)) {
                    status = ST_CONVERGED;
                    active = false;
                } else if (singular) {
                    status = ST_BREAKDOWN;
                    active = false;
                } else if (it >= C.max_iters) {
                    status = ST_MAX_ITER;
                    active = false;
                } else if (estimate_ok && ++restarts > kMaxRestarts) {
                    status = kStagnated;
                    active = false;
                }
            }
        }
    }
    const bool done = folded_finish<FMT, SF>(A, S, as, pb, io, sigma, X, eX, bX, Rv, eR, bR, run && accepted(status), it,
                                             status, true, beta2, tau2, nb2, sm, g, tm);
    // The basis is dead scratch from here on: its whole 128-byte lines are dropped
    // from L2 without a write-back (as gmres_packed_system).
    if (done && V != nullptr) {
        const uintptr_t first = (reinterpret_cast<uintptr_t>(V) + 127) & ~static_cast<uintptr_t>(127);
        const uintptr_t end = (reinterpret_cast<uintptr_t>(V) + (size_t)(m + 1) * vs * 8) & ~static_cast<uintptr_t>(127);
        for (uintptr_t a = first + (uintptr_t)tm.tid * 128; a < end; a += (uintptr_t)tm.nt * 128)
            asm volatile("discard.global.L2 [%0], 128;" ::"l"(a) : "memory");
    }
    return done ? kDone : run ? kLeft : kUnfit;
}

}  // namespace fx
}  // namespace bbs
