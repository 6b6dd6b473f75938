// rng_tables.cpp -- the tables of the device generator's normals (rng.cu).
#include <cmath>

#include "rng_tables.h"

namespace bmf {

// The tables, from long double (host side, once per process).
const GenTables &gen_tables()
{
    static const GenTables *tab = [] {
        GenTables *t = new GenTables;
        for (int i = 0; i < 1024; ++i) {
            const double c = i == 0 ? 1.0 : i == 1023 ? 0.5 : (double)(1.0L / (1.0L + (i + 0.5L) / 1024.0L));
            t->lg[i].c = c;
            t->lg[i].ln = (double)-logl(i >= kLogHalf ? 2.0L * c : (long double)c);
        }
        const long double turn = 6.283185307179586476925286766559005768L / 2048.0L;
        for (int k = 0; k < 512; ++k) {
            const long double s = sinl(turn * k), c = cosl(turn * k);
            SinCos &e = t->sc[k];
            e.s = (double)s;
            e.c = (double)c;
            e.sp[0] = (float)s;
            e.sp[1] = (float)(s - (long double)e.sp[0]);
            e.sp[2] = (float)c;
            e.sp[3] = (float)(c - (long double)e.sp[2]);
        }
        return t;
    }();
    return *tab;
}

}  // namespace bmf
