"""Writes translate_gen.cuh: straight-line M2M / L2L building blocks at fixed order P = 1..6 on one thread's registers.

Multi-indices are ordered by total degree, then nx descending, then ny descending.  A translation by (+-s/4)^3 is
one-dimensional shifts along x, y and z in place, with a[d] = (+-1/4)^d / d!:
  shift_moments_P(v, axis coefficients)  v^n += sum_{1 <= d <= n_e} a[d] v^(n - d e)  (v = M/n!, highest degree first)
  shift_locals_P                         v^n += sum_{1 <= d <= P - |n|} a[d] v^(n + d e)  (lowest degree first)
and the constant factors around them: moments_in (2^-|n| / n!), moments_out (n!), locals_out (2^-(|n| + 1)),
moments_scale (1/n! from the quadrupole on), locals_harmonic (add the n_z <= 1 coefficients h, complete the others).
Run: python gen_translate.py > translate_gen.cuh
"""
from math import factorial

PMAX_GEN = 6


def multi_indices(p):
    return [(nx, ny, o - nx - ny) for o in range(p + 1) for nx in range(o, -1, -1) for ny in range(o - nx, -1, -1)]


def fact(v):
    return factorial(v[0]) * factorial(v[1]) * factorial(v[2])


def main():
    print("// Generated by gen_translate.py -- M2M and L2L building blocks (do not edit).")
    print("#pragma once")
    print()
    print("template <int P> struct XlGen;")
    for P in range(1, PMAX_GEN + 1):
        mi = multi_indices(P)
        idx = {v: i for i, v in enumerate(mi)}
        nc = len(mi)
        H = [k for k in mi if k[2] <= 1]
        fn = "    template <class T> static __device__ __forceinline__ void"
        print(f"template <> struct XlGen<{P}> {{")
        print(f"    static constexpr int NC = {nc};")
        print(f"    static constexpr int NH = {len(H)};")
        for name, up in (("shift_moments", False), ("shift_locals", True)):
            print(f"{fn} {name}(T (&v)[{nc}], const T (&ax)[{P + 1}], const T (&ay)[{P + 1}], const T (&az)[{P + 1}])")
            print("    {")
            for e, a in enumerate(("ax", "ay", "az")):
                for k in (range(nc) if up else range(nc - 1, 0, -1)):
                    v = mi[k]
                    for d in range(1, (P - sum(v) if up else v[e]) + 1):
                        w = list(v)
                        w[e] += d if up else -d
                        print(f"        v[{k}] += {a}[{d}] * v[{idx[tuple(w)]}];")
            print("    }")
        for name, f in (("moments_in", lambda v: f"(T(1) / T({fact(v) << sum(v)}))"), ("moments_out", lambda v: f"T({fact(v)})"),
                        ("locals_out", lambda v: f"(T(1) / T({2 << sum(v)}))")):
            print(f"{fn} {name}(T (&v)[{nc}])")
            print("    {")
            for k, v in enumerate(mi):
                print(f"        v[{k}] *= {f(v)};")
            print("    }")
        print(f"{fn} moments_scale(T (&v)[{nc}])")
        print("    {")
        for k, v in enumerate(mi):
            if k >= 4:
                print(f"        v[{k}] *= T(1) / T({fact(v)});")
        print("    }")
        print(f"{fn} locals_harmonic(T (&v)[{nc}], const T (&h)[{len(H)}])")
        print("    {")
        for k, v in enumerate(mi):
            if v[2] <= 1:
                print(f"        v[{k}] += h[{H.index(v)}];")
            else:
                print(f"        v[{k}] = -v[{idx[(v[0] + 2, v[1], v[2] - 2)]}] - v[{idx[(v[0], v[1] + 2, v[2] - 2)]}];")
        print("    }")
        print("};")


if __name__ == "__main__":
    main()
