// Per-element steps of the classic (Fig. 2) and pipelined (Fig. 4) loops and
// the solver's view of one system (Ctx). The per-solve kernels
// (kernels_solver.cu) and the per-step kernels of the serving engine
// (kernels_step.cu) both compute every element through these functions, so
// the two paths take the same fma forms and give the same bits.
#pragma once

#include "kernels.cuh"

namespace rbs {

constexpr int SQ = 4;  // register-window placements of the SpMV kernels' dots
// The vector kernels' dots: K4 and P1 (a product and a square), P3 (four products
// and a square). Words enough that products stay in the window while the Krylov
// vectors still fall off by orders of magnitude per grid layer (P3 at 192^3, b = A
// 1, second iteration: 313 us with 9 words, 225 with 12; later ones 177 either
// way).
using RowsR2 = ExactRows<2, 14, false>;
using RowsR5 = ExactRows<5, 12, false>;

struct Ctx {
    CSRView A;
    DiagArgs D;  // with the SPMV_MODE_DIAG* schedules
    int64_t n;
    double *x, *r, *r0, *p, *ph, *s, *q, *qh, *y, *invd;
    double *rh, *w, *wh, *t, *sh, *z, *zh, *v;
    const double *b, *x0;
    const double *diag;  // the caller's Jacobi diagonal (per-step path only; null: diag(A))
    SolverState *st;
    DotScratch *g;
    double *hist;
    unsigned *err;
    int spmv_mode;
};

// Two outputs of one element step.
struct VPair {
    double a, b;
};

// set-up, classic: r = RN(b - A x0) (or b), x = x0 (or +0), r0 = p = r,
// phat = RN(r * invd); returns r_i
__device__ __forceinline__ double cls_setup_elem(const Ctx &c, int64_t i, bool &bad) {
    double ri;
    if (c.x0) {
        const double ax = spmv_row(c.A, i, c.x0, bad);
        ri = __dsub_rn(c.b[i], ax);
        c.x[i] = c.x0[i];
    } else {
        ri = c.b[i];
        c.x[i] = 0.0;
    }
    c.r[i] = ri;
    c.r0[i] = ri;
    c.p[i] = ri;
    c.ph[i] = __dmul_rn(ri, c.invd[i]);
    return ri;
}

// S4, S5: q = fma(-alpha, s, r), qhat = RN(q * invd)  -> (q, qhat)
__device__ __forceinline__ VPair cls_k2(double na, double s, double r, double d) {
    const double q = fma(na, s, r);
    return VPair{q, __dmul_rn(q, d)};
}

// S8, S9: x = fma(omega, qhat, fma(alpha, phat, x)), r = fma(-omega, y, q)  -> (x, r)
__device__ __forceinline__ VPair cls_k4(double al, double om, double nom, double qh, double ph, double x, double y,
                                        double q) {
    return VPair{fma(om, qh, fma(al, ph, x)), fma(nom, y, q)};
}

// S12, S1: p = fma(beta, fma(-omega, s, p), r), phat = RN(p * invd)  -> (p, phat)
__device__ __forceinline__ VPair cls_k5(double be, double nom, double s, double p, double r, double d) {
    const double pn = fma(be, fma(nom, s, p), r);
    return VPair{pn, __dmul_rn(pn, d)};
}

// set-up 1, pipelined: r = RN(b - A x0) (or b), x, r0 = r, rhat = RN(r * invd)
__device__ __forceinline__ void pipe_setup1_elem(const Ctx &c, int64_t i, bool &bad) {
    double ri;
    if (c.x0) {
        const double ax = spmv_row(c.A, i, c.x0, bad);
        ri = __dsub_rn(c.b[i], ax);
        c.x[i] = c.x0[i];
    } else {
        ri = c.b[i];
        c.x[i] = 0.0;
    }
    c.r[i] = ri;
    c.r0[i] = ri;
    c.rh[i] = __dmul_rn(ri, c.invd[i]);
}

// P1 for one element: in[0..5] = rh, w, wh, t, r, invd and, after iteration 0,
// in[6..11] = ph, s, sh, z, zh, v (all loaded by the caller before any store);
// out = ph, s, sh, z, q, qh, y, zh.
struct P1In {
    double rh, w, wh, t, r, d, ph, s, sh, z, zh, v;
};
struct P1Out {
    double ph, s, sh, z, q, qh, y, zh;
};
__device__ __forceinline__ P1Out p1_step(const P1In &a, bool first, double nal, double be, double nom) {
    P1Out o;
    if (first) {
        o.ph = a.rh;
        o.s = a.w;
        o.sh = a.wh;
        o.z = a.t;
    } else {
        o.ph = fma(be, fma(nom, a.sh, a.ph), a.rh);
        o.s = fma(be, fma(nom, a.z, a.s), a.w);
        o.sh = fma(be, fma(nom, a.zh, a.sh), a.wh);
        o.z = fma(be, fma(nom, a.v, a.z), a.t);
    }
    o.q = fma(nal, o.s, a.r);
    o.qh = fma(nal, o.sh, a.rh);
    o.y = fma(nal, o.z, a.w);
    o.zh = __dmul_rn(o.z, a.d);
    return o;
}
// with its dots' products
template <class R>
__device__ __forceinline__ P1Out p1_elem(const P1In &a, bool first, double nal, double be, double nom, R &red) {
    const P1Out o = p1_step(a, first, nal, be, nom);
    red.add(0, o.q, o.y);
    red.add_sq(1, o.y);
    return o;
}

__device__ __forceinline__ P1In p1_load(const Ctx &c, int64_t i, bool first) {
    P1In a{c.rh[i], c.w[i], c.wh[i], c.t[i], c.r[i], c.invd[i], 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (!first) {
        a.ph = c.ph[i];
        a.s = c.s[i];
        a.sh = c.sh[i];
        a.z = c.z[i];
        a.zh = c.zh[i];
        a.v = c.v[i];
    }
    return a;
}

__device__ __forceinline__ void p1_store(const Ctx &c, int64_t i, const P1Out &o) {
    c.ph[i] = o.ph;
    c.s[i] = o.s;
    c.sh[i] = o.sh;
    c.z[i] = o.z;
    c.q[i] = o.q;
    c.qh[i] = o.qh;
    c.y[i] = o.y;
    c.zh[i] = o.zh;
}

// P3 for one element, from its thirteen operands (loaded by the caller before
// any store): x, r, rhat, w and what, and the five dots' products.
struct P3In {
    double qh, y, q, ph, x, zh, wh, v, t, d, r0, s, z;
};
struct P3Out {
    double x, r, rh, w, wh;
};
__device__ __forceinline__ P3Out p3_step(const P3In &a, double al, double nal, double om, double nom) {
    P3Out o;
    o.x = fma(om, a.qh, fma(al, a.ph, a.x));
    o.r = fma(nom, a.y, a.q);
    o.rh = fma(nom, fma(nal, a.zh, a.wh), a.qh);
    o.w = fma(nom, fma(nal, a.v, a.t), a.y);
    o.wh = __dmul_rn(o.w, a.d);
    return o;
}
// with its dots' products
template <class R>
__device__ __forceinline__ P3Out p3_elem(const P3In &a, double al, double nal, double om, double nom, R &red) {
    const P3Out o = p3_step(a, al, nal, om, nom);
    red.add(0, a.r0, o.r);
    red.add(1, a.r0, o.w);
    red.add(2, a.r0, a.s);
    red.add(3, a.r0, a.z);
    red.add_sq(4, o.r);
    return o;
}

// ---- the vector steps with dots over a range of element pairs ---------------------
//
// Pairs first, first + step, ... below end (element 2j and 2j + 1 of pair j, with
// 16-byte accesses), then the odd last element `odd` (< 0: none) in the thread
// that has one. Every operand is loaded before the first store (the vectors are
// not restrict-qualified, so later loads could not be issued early). The first
// turn is taken by every thread of the block, with or without a pair, since the
// reducer's windows open on the block's first products.

template <class R, class F>
__device__ __forceinline__ void each_pair(int64_t first, int64_t end, int64_t step, F &&f) {
    bool open = R::WINDOWS;
    for (int64_t j = first;; j += step) {
        const bool live = j < end;
        if (!live && !open) break;
        f(2 * j, live, open);
        open = false;
        if (!live) break;
    }
}

__device__ __forceinline__ double2 ld2_if(bool live, const double *p, int64_t i) {
    return live ? ld2(p, i) : make_double2(0.0, 0.0);
}

// K4: x, r, <r0,r>, <r,r>
template <class R>
__device__ __forceinline__ void cls_k4_pairs(const Ctx &c, R &red, double al, double om, int64_t first, int64_t end,
                                             int64_t step, int64_t odd) {
    const double nom = -om;
    each_pair<R>(first, end, step, [&](int64_t i, bool live, bool open) {
        const double2 qh = ld2_if(live, c.qh, i), ph = ld2_if(live, c.ph, i), y = ld2_if(live, c.y, i),
                      q = ld2_if(live, c.q, i), r0 = ld2_if(live, c.r0, i), x = ld2_if(live, c.x, i);
        const VPair u0 = cls_k4(al, om, nom, qh.x, ph.x, x.x, y.x, q.x);
        const VPair u1 = cls_k4(al, om, nom, qh.y, ph.y, x.y, y.y, q.y);
        if (open)
            red.open({max(R::limb_of(r0.x, u0.b), R::limb_of(r0.y, u1.b)),
                      max(R::limb_of(u0.b, u0.b), R::limb_of(u1.b, u1.b))});
        if (live) {
            st2(c.x, i, make_double2(u0.a, u1.a));
            st2(c.r, i, make_double2(u0.b, u1.b));
            const double a0[2] = {r0.x, r0.y}, r[2] = {u0.b, u1.b};
            red.template add<2>(0, a0, r);
            red.template add_sq<2>(1, r);
        }
    });
    if (odd >= 0) {
        const VPair u = cls_k4(al, om, nom, c.qh[odd], c.ph[odd], c.x[odd], c.y[odd], c.q[odd]);
        c.x[odd] = u.a;
        c.r[odd] = u.b;
        red.add(0, c.r0[odd], u.b);
        red.add_sq(1, u.b);
    }
}

// P1: S1-S7, S9, <q,y>, <y,y>
template <class R>
__device__ __forceinline__ void pipe_p1_pairs(const Ctx &c, R &red, bool it0, double nal, double be, double nom,
                                              int64_t first, int64_t end, int64_t step, int64_t odd) {
    each_pair<R>(first, end, step, [&](int64_t i, bool live, bool open) {
        const double2 rh = ld2_if(live, c.rh, i), w = ld2_if(live, c.w, i), wh = ld2_if(live, c.wh, i),
                      t = ld2_if(live, c.t, i), r = ld2_if(live, c.r, i), d = ld2_if(live, c.invd, i);
        const bool old = live && !it0;
        const double2 ph = ld2_if(old, c.ph, i), s = ld2_if(old, c.s, i), sh = ld2_if(old, c.sh, i),
                      z = ld2_if(old, c.z, i), zh = ld2_if(old, c.zh, i), v = ld2_if(old, c.v, i);
        const P1Out o0 =
            p1_step(P1In{rh.x, w.x, wh.x, t.x, r.x, d.x, ph.x, s.x, sh.x, z.x, zh.x, v.x}, it0, nal, be, nom);
        const P1Out o1 =
            p1_step(P1In{rh.y, w.y, wh.y, t.y, r.y, d.y, ph.y, s.y, sh.y, z.y, zh.y, v.y}, it0, nal, be, nom);
        if (open)
            red.open({max(R::limb_of(o0.q, o0.y), R::limb_of(o1.q, o1.y)),
                      max(R::limb_of(o0.y, o0.y), R::limb_of(o1.y, o1.y))});
        if (live) {
            st2(c.ph, i, make_double2(o0.ph, o1.ph));
            st2(c.s, i, make_double2(o0.s, o1.s));
            st2(c.sh, i, make_double2(o0.sh, o1.sh));
            st2(c.z, i, make_double2(o0.z, o1.z));
            st2(c.q, i, make_double2(o0.q, o1.q));
            st2(c.qh, i, make_double2(o0.qh, o1.qh));
            st2(c.y, i, make_double2(o0.y, o1.y));
            st2(c.zh, i, make_double2(o0.zh, o1.zh));
            const double q[2] = {o0.q, o1.q}, y[2] = {o0.y, o1.y};
            red.template add<2>(0, q, y);
            red.template add_sq<2>(1, y);
        }
    });
    if (odd >= 0) p1_store(c, odd, p1_elem(p1_load(c, odd, it0), it0, nal, be, nom, red));
}

// P3: S12-S15, S17, <r0,r>, <r0,w>, <r0,s>, <r0,z>, <r,r>
template <class R>
__device__ __forceinline__ void pipe_p3_pairs(const Ctx &c, R &red, double al, double om, int64_t first, int64_t end,
                                              int64_t step, int64_t odd) {
    const double nal = -al, nom = -om;
    each_pair<R>(first, end, step, [&](int64_t i, bool live, bool open) {
        const double2 qh = ld2_if(live, c.qh, i), y = ld2_if(live, c.y, i), q = ld2_if(live, c.q, i),
                      ph = ld2_if(live, c.ph, i), x = ld2_if(live, c.x, i), zh = ld2_if(live, c.zh, i),
                      wh = ld2_if(live, c.wh, i), v = ld2_if(live, c.v, i), t = ld2_if(live, c.t, i),
                      d = ld2_if(live, c.invd, i), r0 = ld2_if(live, c.r0, i), s = ld2_if(live, c.s, i),
                      z = ld2_if(live, c.z, i);
        const P3Out o0 = p3_step(P3In{qh.x, y.x, q.x, ph.x, x.x, zh.x, wh.x, v.x, t.x, d.x, r0.x, s.x, z.x}, al, nal, om, nom);
        const P3Out o1 = p3_step(P3In{qh.y, y.y, q.y, ph.y, x.y, zh.y, wh.y, v.y, t.y, d.y, r0.y, s.y, z.y}, al, nal, om, nom);
        if (open)
            red.open({max(R::limb_of(r0.x, o0.r), R::limb_of(r0.y, o1.r)),
                      max(R::limb_of(r0.x, o0.w), R::limb_of(r0.y, o1.w)),
                      max(R::limb_of(r0.x, s.x), R::limb_of(r0.y, s.y)),
                      max(R::limb_of(r0.x, z.x), R::limb_of(r0.y, z.y)),
                      max(R::limb_of(o0.r, o0.r), R::limb_of(o1.r, o1.r))});
        if (live) {
            st2(c.x, i, make_double2(o0.x, o1.x));
            st2(c.r, i, make_double2(o0.r, o1.r));
            st2(c.rh, i, make_double2(o0.rh, o1.rh));
            st2(c.w, i, make_double2(o0.w, o1.w));
            st2(c.wh, i, make_double2(o0.wh, o1.wh));
            const double a0[2] = {r0.x, r0.y}, r[2] = {o0.r, o1.r}, w[2] = {o0.w, o1.w}, sv[2] = {s.x, s.y},
                         zv[2] = {z.x, z.y};
            red.template add<2>(0, a0, r);
            red.template add<2>(1, a0, w);
            red.template add<2>(2, a0, sv);
            red.template add<2>(3, a0, zv);
            red.template add_sq<2>(4, r);
        }
    });
    if (odd >= 0) {
        const P3Out o = p3_elem(P3In{c.qh[odd], c.y[odd], c.q[odd], c.ph[odd], c.x[odd], c.zh[odd], c.wh[odd],
                                     c.v[odd], c.t[odd], c.invd[odd], c.r0[odd], c.s[odd], c.z[odd]},
                                al, nal, om, nom, red);
        c.x[odd] = o.x;
        c.r[odd] = o.r;
        c.rh[odd] = o.rh;
        c.w[odd] = o.w;
        c.wh[odd] = o.wh;
    }
}

}  // namespace rbs
