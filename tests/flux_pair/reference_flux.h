// The kinetic split flux from the q-variables, evaluated directly in type R:
// binary128 (Real) as the reference, or double.
#pragma once

#include <cmath>

#ifdef __x86_64__
#include <quadmath.h>
using Real = __float128;
static Real Exp(Real x) { return expq(x); }
static Real Log(Real x) { return logq(x); }
static Real Sqrt(Real x) { return sqrtq(x); }
static Real Erfc(Real x) { return erfcq(x); }
#else  // long double is binary128
using Real = long double;
static Real Exp(Real x) { return std::exp(x); }
static Real Log(Real x) { return std::log(x); }
static Real Sqrt(Real x) { return std::sqrt(x); }
static Real Erfc(Real x) { return std::erfc(x); }
#endif
static double Exp(double x) { return std::exp(x); }
static double Log(double x) { return std::log(x); }
static double Sqrt(double x) { return std::sqrt(x); }
static double Erfc(double x) { return std::erfc(x); }

template <class R>
static void flux(const R q[4], int axis, int sign, R G[4]) {
    const R beta = -q[3] / 2, u = q[1] / (2 * beta), v = q[2] / (2 * beta), uu = u * u + v * v;
    const R rho = Exp(q[0] - Log(beta) * R(2.5) + beta * uu), p = rho / (2 * beta);
    const R a = axis ? v : u, b = axis ? u : v, E = p * R(2.5) + rho * uu / 2, sb = Sqrt(beta);
    const R S = a * sb, A = Erfc(-sign * S) / 2;
    const R pi = R(0x1.921fb54442d18p+1) + R(0x1.1a62633145c07p-53);
    const R B = sign * Exp(-S * S) / (2 * Sqrt(pi) * sb);
    G[0] = rho * (a * A + B);
    G[1] = (p + rho * a * a) * A + rho * a * B;
    G[2] = b * G[0];
    G[3] = (p + E) * a * A + (E + p / 2) * B;
}
