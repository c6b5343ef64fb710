// cos_poly.h -- written by gen_cos_poly.py; do not edit.
// cos(d) ~= sum_k C_k (d^2)^k for d in [0, pi] (Lawson minimax fits):
// COS_C: degree 6 in d^2, max error in FP32 evaluation 6.15e-07;
// COS5_C: degree 5 in d^2, max error in FP32 evaluation 1.27e-06;
// sin(d) ~= d * sum_k S_k (d^2)^k for d in [0, pi]:
// SIN5_C: degree 5 in d^2, max error in FP32 evaluation 4.44e-07.
// sin(pi/2 x) ~= x * sum_k QSIN_C_k (x^2)^k and cos(pi/2 x) ~= sum_k QCOS_C_k
// (x^2)^k for |x| <= 1/2: max error in FP32 8.32e-08 and 5.51e-08.
#pragma once

namespace cgh {

constexpr float COS_C0 = 1.0f;
constexpr float COS_C1 = -0.49999991059303284f;
constexpr float COS_C2 = 0.04166649281978607f;
constexpr float COS_C3 = -0.001388781820423901f;
constexpr float COS_C4 = 2.477006273693405e-05f;
constexpr float COS_C5 = -2.707994326556218e-07f;
constexpr float COS_C6 = 1.7246171157836443e-09f;

constexpr float COS5_C0 = 0.9999993443489075f;
constexpr float COS5_C1 = -0.49999457597732544f;
constexpr float COS5_C2 = 0.04165996238589287f;
constexpr float COS5_C3 = -0.0013859154423698783f;
constexpr float COS5_C4 = 2.420584496576339e-05f;
constexpr float COS5_C5 = -2.1980551423439465e-07f;

constexpr float SIN5_C0 = 0.9999996423721313f;
constexpr float SIN5_C1 = -0.16666558384895325f;
constexpr float SIN5_C2 = 0.008332425728440285f;
constexpr float SIN5_C3 = -0.00019809025980066508f;
constexpr float SIN5_C4 = 2.700008735700976e-06f;
constexpr float SIN5_C5 = -2.037002744259553e-08f;

constexpr float QSIN_C0 = 1.5707963705062866f;
constexpr float QSIN_C1 = -0.6459634900093079f;
constexpr float QSIN_C2 = 0.07968010008335114f;
constexpr float QSIN_C3 = -0.004601663444191217f;

constexpr float QCOS_C0 = 1.0f;
constexpr float QCOS_C1 = -1.2337005138397217f;
constexpr float QCOS_C2 = 0.25366923213005066f;
constexpr float QCOS_C3 = -0.020860297605395317f;
constexpr float QCOS_C4 = 0.0009040222503244877f;

}  // namespace cgh
