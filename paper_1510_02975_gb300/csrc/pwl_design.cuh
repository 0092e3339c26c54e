// pwl_design.cuh -- internal interface of the batched design and projection
// kernels (one function is a batch of one).
#pragma once

#include "pwl_common.cuh"

namespace pwl {

constexpr int kMaxIntervals = 1048575;

// 1/d for a positive normal FP64 d from the hardware's approximate reciprocal
// (rcp.approx.ftz.f64, relative error e below 2^-19.9) by one step of third
// order, r (1 + e + e^2) with e = 1 - d r: what remains, e^3, is below FP64
// rounding.  Three FP64 operations against about ten for a division (the Gram
// solves and the table build's slopes and reciprocal lengths).
__device__ __forceinline__ double recip_newton(double d)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// F functions; function f owns knots koff[f] .. koff[f+1]-1 (N_f + 1 of them),
// density cells moff[f] .. moff[f+1]-1 (M_f) and chunks choff[f] .. choff[f+1]-1.
// Which kinds a plan holds: the hot kernels are compiled once for the
// analytic kinds and once for sampled functions (whose FP64 interpolation
// would otherwise weigh on the analytic loops' registers); a launch runs the
// instantiations its plan needs.  0 means both.
constexpr int kKindsAnalytic = 1;
constexpr int kKindsSampled = 2;
inline int plan_kinds(int kinds) { return kinds ? kinds : (kKindsAnalytic | kKindsSampled); }
inline int kinds_of(const pwl_func* f, int64_t n)
{
    int k = 0;
    for (int64_t i = 0; i < n; ++i) k |= f[i].kind == PWL_F_SAMPLED ? kKindsSampled : kKindsAnalytic;
    return k;
}

// A function's constants in the FP32 mode of a batch
struct DesignFunc {
    FuncF g;
    float deltaf;     // cell width, rounded
    double a, delta;  // interval start, cell width
    double cunit;     // G_M / (N delta): tau_i / delta = i cunit (0: the uniform partition)
};

struct DesignPlan {
    int F;
    int precision;
    int kinds;  // kKindsAnalytic | kKindsSampled of the functions (0: both)
    const pwl_func* funcs;
    const int64_t* koff;
    const int64_t* moff;
    const int64_t* choff;
    int64_t n_max;         // the most intervals of a function
    int64_t total_knots, total_cells, total_chunks;
    const double* delta;   // F cell widths (b - a) / M
    const int* tile_func;  // per tile of 8 chunks: its function (NULL: one function)
    DesignFunc* ffuncs;    // FP32 mode of a batch: F constants (scratch)
    double* d;       // total_cells densities (FP32 mode of a batch: floats, every function 16-byte aligned)
    double* csum;    // total_chunks partial sums
    double* cbase;   // total_chunks exclusive chunk bases
    int64_t* plast;  // per chunk: its last cell of positive density, then (after the scan) the last one before
                     // it, or -1
    double* stot;    // per function: G_M = delta sum d (not in the FP32 mode of a batch)
    double* knots;   // total_knots output
};

int64_t design_chunks(int64_t M);
size_t design_scratch_bytes(int64_t F, int64_t total_cells, int64_t total_chunks);
void design_carve_scratch(DesignPlan& p, void* scratch);
pwl_status design_launch(const DesignPlan& p, cudaStream_t s);
// FP32 mode of a batch; needs p.tile_func and p.ffuncs.
pwl_status design_batch_f_launch(const DesignPlan& p, cudaStream_t s);

// Projection: F functions with knots at koff (device), values out.
struct ProjectPlan {
    int F;
    int precision;
    int kinds;  // kKindsAnalytic | kKindsSampled of the functions (0: both)
    int form;
    int max_rows;          // max over f of N_f + 1
    int64_t total_knots;
    int64_t total_intervals;
    const pwl_func* funcs;
    const FuncValueF* funcs_f;  // the functions' FP32 parameters (FP32 mode of P_T)
    const int64_t* koff;
    const double* knots;
    double* values;
    double2* lr;           // per interval: (int f phi_left, int f phi_right)
    double* cr;            // solver scratch: 4 doubles per knot (and 128 per function of several)
    int solver;            // 0: cyclic reduction, one CTA per function; 1: partitioned Thomas, one warp per function
    const int* order;      // solver 1: the order in which warps take the functions (NULL: 0..F-1)
};

struct GaussLegendre {
    int Q;
    double x[16];   // nodes on [-1, 1]
    double w[16];   // weights
    double wl[16];  // w (1 - x) / 2: the weight times the left hat phi_{j-1} at the node
    double wr[16];  // w (1 + x) / 2: the weight times the right hat phi_j at the node
    float xf[16];   // nodes rounded to FP32
    float wlh[16], wll[16], wrh[16], wrl[16];  // wl, wr split into FP32 pairs hi + lo
};
const GaussLegendre& gauss_legendre_rule(int Q);

size_t project_scratch_bytes(int64_t total_knots, int64_t total_intervals);
void project_carve_scratch(ProjectPlan& p, void* scratch);
pwl_status project_launch(const ProjectPlan& p, const GaussLegendre& gl, cudaStream_t s);

}  // namespace pwl
