"""Generate one CUDA translation unit per angular class pair of the
real-space kernels (real_q<cb><ck>.cu), so that the 21 instantiations
compile in parallel.  Run from this directory: python gen_units.py"""
CLASSES = [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2)]

# Which kernel runs a class pair (NV elements in its Cartesian block, L its
# total momentum):
#   * one warp per bra with its stages refilled (k_real_w, real2.cuh) while a
#     lane can hold the block: NV <= 36 in FP32, NV <= 27 in FP64;
#   * one warp per image quartet (k_real_c, real3.cuh) above that.
# The FP64 list pass takes k_real_list_w up to NV = 36 and k_real_list_c above.
# Class pairs of s and p shells have two more tile-kernel families, the
# lane-per-bra kernels of kernels.cuh and the pair-queue kernels of real2.cuh,
# and the autotuner picks one per class pair (RealLaunch::variant).
ARGS32 = "a.pl, a.b0, a.b1, a.k0, a.k1, a.same, a.kchunk, a.mode, a.tau, a.Dpf, a.dmaxf, a.X, a.Y, a.cnt, a.big, a.nbig, a.cap, a.ovf"
ARGSW32 = ARGS32.replace("a.b0, a.b1, a.k0, a.k1, a.same, a.kchunk", "a.map, a.k0, a.k1, a.same")
ARGSW64 = ARGSW32.replace("a.Dpf, a.dmaxf", "a.Dp, a.dmax")
ARGS64 = ARGS32.replace("a.Dpf, a.dmaxf", "a.Dp, a.dmax")

HEAD = """// Real-space quartet kernels for bra class {lab} and ket class {lcd} (generated by gen_units.py).
{jeng}#include "launch.h"
#include "real3.cuh"

namespace jk {{

void launch_real_q{cb}{ck}(const RealLaunch &a)
{{
    const int nb = a.b1 - a.b0, nk = a.k1 - a.k0;
    if (nb <= 0 || nk <= 0) return;
    if (a.list_pass) {{
        {list};
        return;
    }}
"""

FAMILIES = """    const dim3 tile((nb + kRealThreads - 1) / kRealThreads, (nk + a.kchunk - 1) / a.kchunk);
    if (a.variant == 2) {{
        if (a.fp32)
            k_real_q<{q}, float><<<tile, kRealThreads, 0, a.st>>>({args32});
        else
            k_real_q<{q}, double><<<tile, kRealThreads, 0, a.st>>>({args64});
        return;
    }}
    if (a.variant == 0) {{
        if (a.fp32)
            k_real<{q}, float><<<tile, kRealThreads, 0, a.st>>>({args32});
        else
            k_real<{q}, double><<<tile, kRealThreads, 0, a.st>>>({args64});
        return;
    }}
"""

TAIL = """    if (a.map.items <= 0) return;
    if (a.fp32)
        {k32}({argsw32});
    else
        {k64}({argsw64});
}}
"""

# Coulomb-only builds take the J-engine where both sides have a d shell (kJengClass in build.cu)
JENG = """
void launch_jeng_q{cb}{ck}(const RealLaunch &a)
{{
    const int nb = a.b1 - a.b0, nk = a.k1 - a.k0;
    if (nb <= 0 || nk <= 0) return;
    dim3 grid((nb + kRealThreads - 1) / kRealThreads, (nk + a.kchunk - 1) / a.kchunk);
    if (a.fp32)
        k_jeng<{q}, float><<<grid, kRealThreads, 0, a.st>>>(a.pl, a.b0, a.b1, a.k0, a.k1, a.same, a.kchunk, a.mode, a.tau, a.dmaxf, a.DhF, a.hs,
                                                            a.X, a.JH, a.cnt, a.big, a.nbig, a.cap, a.ovf);
    else
        k_jeng<{q}, double><<<grid, kRealThreads, 0, a.st>>>(a.pl, a.b0, a.b1, a.k0, a.k1, a.same, a.kchunk, a.mode, a.tau, a.dmax, a.DhD, a.hs,
                                                             a.X, a.JH, a.cnt, a.big, a.nbig, a.cap, a.ovf);
}}
"""

END = """
}}  // namespace jk
"""


def ncart(l):
    return (l + 1) * (l + 2) // 2


def unit(cb, ck):
    la, lb = CLASSES[cb]
    lc, ld = CLASSES[ck]
    nv = ncart(la) * ncart(lb) * ncart(lc) * ncart(ld)
    q = "%d, %d, %d, %d" % (la, lb, lc, ld)

    def tile(t, lim):
        if nv <= lim:
            return "k_real_w<%s, %s><<<(unsigned)((a.map.items + kWarpsPerBlock - 1) / kWarpsPerBlock), 32 * kWarpsPerBlock, 0, a.st>>>" % (q, t)
        return "k_real_c<%s, %s><<<(unsigned)a.map.items, 32, 0, a.st>>>" % (q, t)

    lst = "(a.pl, a.big, a.nbig, a.cap, a.same, a.Dp, a.X, a.Y, a.cnt64)"
    if nv <= 36:
        lst = "k_real_list_w<%s><<<152 * 8, 32 * kWarpsPerBlock, 0, a.st>>>%s" % (q, lst)
    else:
        lst = "k_real_list_c<%s><<<152 * 16, 32, 0, a.st>>>%s" % (q, lst)
    body = HEAD + (FAMILIES if max(la, lb, lc, ld) <= 1 else "") + TAIL + (JENG if cb >= 3 else "") + END
    return body.format(cb=cb, ck=ck, lab=(la, lb), lcd=(lc, ld), q=q, list=lst, jeng='#include "jeng.cuh"\n' if cb >= 3 else "", k32=tile("float", 36), k64=tile("double", 27),
                       args32=ARGS32, args64=ARGS64, argsw32=ARGSW32, argsw64=ARGSW64)


def main():
    decls = []
    for cb in range(len(CLASSES)):
        for ck in range(cb, len(CLASSES)):
            open("real_q%d%d.cu" % (cb, ck), "w").write(unit(cb, ck))
            decls.append((cb, ck))
    with open("real_units.h", "w") as f:
        f.write("// Declarations of the per-class-pair launchers (generated by gen_units.py).\n#pragma once\n#include \"launch.h\"\n\n")
        f.write("namespace jk {\n")
        for cb, ck in decls:
            f.write("void launch_real_q%d%d(const RealLaunch &a);\n" % (cb, ck))
            if cb >= 3:
                f.write("void launch_jeng_q%d%d(const RealLaunch &a);\n" % (cb, ck))
        f.write("\n// class pairs of s and p shells have the lane-per-bra and pair-queue kernels as further families\n")
        f.write("inline bool real_has_warp_kernel(int cb, int ck) { return cb <= 2 && ck <= 2; }\n")
        f.write("\ninline void launch_real(int cb, int ck, const RealLaunch &a)\n{\n    switch (cb * 8 + ck) {\n")
        for cb, ck in decls:
            f.write("    case %d: launch_real_q%d%d(a); break;\n" % (cb * 8 + ck, cb, ck))
        f.write("    default: break;\n    }\n}\n\n")
        f.write("// Coulomb-only builds: the J-engine kernel of a class pair (jeng.cuh)\n")
        f.write("inline void launch_jeng(int cb, int ck, const RealLaunch &a)\n{\n    switch (cb * 8 + ck) {\n")
        for cb, ck in [d for d in decls if d[0] >= 3]:
            f.write("    case %d: launch_jeng_q%d%d(a); break;\n" % (cb * 8 + ck, cb, ck))
        f.write("    default: break;\n    }\n}\n\n}  // namespace jk\n")


if __name__ == "__main__":
    main()
