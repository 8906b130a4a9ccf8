// Smoothed-aggregation multigrid hierarchy (host side), used as the
// preconditioner of the Poisson-kernel solve.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

// CSR matrix with FP64 values (rows ascending, columns ascending in a row)
struct AmgCsr {
    int64_t rows = 0, cols = 0;
    std::vector<int64_t> off;
    std::vector<int32_t> col;
    std::vector<double> val;
};

// One level: its operator A, the inverse diagonal, the Jacobi weight omega
// (also the prolongator-smoothing weight) and, except on the coarsest level,
// the prolongator P to it from the next coarser level and R = P^T.
//
// With one Jacobi sweep before and after the coarse correction, and the
// prolongator smoothed with the same weight, the level's V-cycle z = V(b) is
//   b_c = Q^T b,   z = G b + Q V_c(b_c),
//   Q = (I - w D^-1 A) P,   G = w D^-1 (2 I - A w D^-1)
// (write S = I - w D^-1 A; the sweep before gives x = w D^-1 b with residual
// S^T b, the coarse right-hand side is P^T S^T b = Q^T b, and the sweep after
// turns x + P e into S x + Q e + w D^-1 b): two sparse products a level
// instead of seven passes.
struct AmgLevel {
    AmgCsr A, P, R, Q, Qt, G;
    std::vector<double> dinv;
    double omega = 0.0;
};

struct AmgHierarchy {
    std::vector<AmgLevel> levels;      // levels[0] is the fine operator
    std::vector<double> coarse_inv;    // dense inverse of the coarsest operator, row-major
    int64_t coarse_n = 0;
};

// Build the hierarchy for the SPD matrix A0; false (with a message) when a
// step fails.  rho0: the finest level's spectral radius of D^-1 A where the
// caller has it (the power iteration's result), else 0.
bool build_amg(const AmgCsr &A0, AmgHierarchy &H, std::string &err, double rho0 = 0.0);

// The device solver's multigrid-preconditioned CG for one right-hand side, on
// the host (a check of the hierarchy and the V-cycle without a GPU): solves
// A x = b to ||r|| <= rtol ||b||.  *levels: hierarchy depth.
bool amg_host_solve(const AmgCsr &A, const std::vector<double> &b, std::vector<double> &x, double rtol,
                    int32_t max_iter, int32_t *iters, int32_t *levels, std::string &err);
