// Generated by gelu_train_fit.py: S(a) = erfcx(a / sqrt 2) / 2 ~ sum_k c_k u^k,
// u = a / 3 - 1, a in [0, 6] (degree 13, weighted least squares).
#pragma once
#define GELU_T_DEG 13
#define GELU_T_COEFFS {1.215139404e-01f, -1.032022983e-01f, 8.240173757e-02f, -6.234495342e-02f, 4.534141719e-02f, -3.103614226e-02f, 1.825407520e-02f, -1.897177473e-02f, 1.077266410e-02f, 1.440767013e-02f, 1.941388473e-02f, -1.222755015e-02f, -2.170337550e-02f, -1.063060481e-02f}
