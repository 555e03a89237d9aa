// One term of the Chebyshev recurrence for one complex entry, shared by the
// kernels that update after a stored application (sg_server.cu) and within one
// (sg_rows.cu): the operations are written out so that both give the same bits.
#pragma once

#include "sg_internal.h"

namespace sg {

// (-i)^q (tr + i ti)
static __device__ __forceinline__ void cheb_rot(int q, double tr, double ti, double &outr, double &outi)
{
    switch (q & 3) {
        case 0: outr = tr; outi = ti; break;
        case 1: outr = ti; outi = -tr; break;
        case 2: outr = -tr; outi = -ti; break;
        default: outr = -ti; outi = tr; break;
    }
}

// x = T_{kn-1}, y = H x, p = T_{kn-2} (unused for kn = 1), a = partial sum
// (formed from x for kn = 1).  Leaves T_kn in p and the sum in a, or, on the
// step's last term, the new psi in p (true: a is not needed any more).
static __device__ __forceinline__ bool cheb_entry(const ChebTerm &t, double xr, double xi, double yr, double yi,
                                                  double &pr, double &pi, double &ar, double &ai)
{
    const double hr = __dmul_rn(fma(-t.ebar, xr, yr), t.inv_de), hi = __dmul_rn(fma(-t.ebar, xi, yi), t.inv_de);
    double tr = hr, ti = hi;
    if (t.kn == 1) {
        ar = __dmul_rn(t.c0, xr);
        ai = __dmul_rn(t.c0, xi);
    } else {
        tr = fma(2.0, hr, -pr);
        ti = fma(2.0, hi, -pi);
    }
    double qr, qi;
    cheb_rot(t.kn, tr, ti, qr, qi);
    ar = fma(t.cn, qr, ar);
    ai = fma(t.cn, qi, ai);
    if (t.kn == t.K) {
        pr = fma(t.cph, ar, -__dmul_rn(t.sph, ai));
        pi = fma(t.sph, ar, __dmul_rn(t.cph, ai));
        return true;
    }
    pr = tr;
    pi = ti;
    return false;
}

// The term that a request's device state stands at.
static __device__ __forceinline__ ChebTerm cheb_term(const ChebState &s)
{
    return ChebTerm{s.k + 1, s.K, s.ebar, s.inv_de, s.cph, s.sph, s.c[0], s.c[s.k + 1]};
}

}  // namespace sg
