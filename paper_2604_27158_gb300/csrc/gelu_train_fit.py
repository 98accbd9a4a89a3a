"""Writes gelu_train_poly.cuh: the polynomial behind the training kernels' GELU and its
derivative, to FP32 accuracy (gelu_fit.py fits the shorter one of the bfloat16 inference).

With a = |v|: Q(a) = Phi(-a) = exp(-a^2 / 2) S(a), S(a) = erfcx(a / sqrt 2) / 2 smooth, fitted by
a polynomial of degree 13 in u = a / 3 - 1 on a in [0, 6] (least squares at Chebyshev nodes,
weight exp(-a^2 / 2) max(a, 1/2): the absolute error of a Q(a), below 5e-9).

Run:  python gelu_train_fit.py > gelu_train_poly.cuh     (needs numpy and scipy)
"""
import numpy as np
from numpy.polynomial import chebyshev as C
from scipy.special import erfcx

DEG, A, NODES = 13, 6.0, 8000


def coefficients():
    u = np.cos(np.pi * (np.arange(NODES) + 0.5) / NODES)
    a = (u + 1.0) * A / 2.0
    w = np.exp(-a * a / 2.0) * np.maximum(a, 0.5)
    c = C.chebfit(u, 0.5 * erfcx(a / np.sqrt(2.0)), DEG, w=w)
    return C.cheb2poly(c).astype(np.float32)


def main():
    print("// Generated by gelu_train_fit.py: S(a) = erfcx(a / sqrt 2) / 2 ~ sum_k c_k u^k,")
    print(f"// u = a / 3 - 1, a in [0, {A:g}] (degree {DEG}, weighted least squares).")
    print("#pragma once")
    print(f"#define GELU_T_DEG {DEG}")
    print(f"#define GELU_T_COEFFS {{{', '.join(f'{float(x):.9e}f' for x in coefficients())}}}")


if __name__ == "__main__":
    main()
