// Real-space quartet kernels for bra class (0, 0) and ket class (2, 2) (generated by gen_units.py).
#include "launch.h"
#include "real3.cuh"

namespace jk {

void launch_real_q05(const RealLaunch &a)
{
    const int nb = a.b1 - a.b0, nk = a.k1 - a.k0;
    if (nb <= 0 || nk <= 0) return;
    if (a.list_pass) {
        k_real_list_w<0, 0, 2, 2><<<152 * 8, 32 * kWarpsPerBlock, 0, a.st>>>(a.pl, a.big, a.nbig, a.cap, a.same, a.Dp, a.X, a.Y, a.cnt64);
        return;
    }
    if (a.map.items <= 0) return;
    if (a.fp32)
        k_real_w<0, 0, 2, 2, float><<<(unsigned)((a.map.items + kWarpsPerBlock - 1) / kWarpsPerBlock), 32 * kWarpsPerBlock, 0, a.st>>>(a.pl, a.map, a.k0, a.k1, a.same, a.mode, a.tau, a.Dpf, a.dmaxf, a.X, a.Y, a.cnt, a.big, a.nbig, a.cap, a.ovf);
    else
        k_real_c<0, 0, 2, 2, double><<<(unsigned)a.map.items, 32, 0, a.st>>>(a.pl, a.map, a.k0, a.k1, a.same, a.mode, a.tau, a.Dp, a.dmax, a.X, a.Y, a.cnt, a.big, a.nbig, a.cap, a.ovf);
}

}  // namespace jk
