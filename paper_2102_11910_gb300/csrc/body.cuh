// Internal definitions of the immersed-body path (body.cu).
#pragma once
#include "common.cuh"

struct pf_schur_s {
    pf_plan plan = nullptr;
    int ns = 0;
    double* x = nullptr;      // surface points (device, ns)
    double* y = nullptr;
    double* ds = nullptr;
    int* six = nullptr;       // smoothed three-point stencils: node indices and weights (ns x 4)
    int* siy = nullptr;
    double* swx = nullptr;
    double* swy = nullptr;
    double* S = nullptr;      // Schur complement, row-major ns x ns
    double* A = nullptr;      // Gauss-Jordan workspace ns x 2 ns
    double* Sinv = nullptr;   // S^-1
    double* f0 = nullptr;     // S^-1 1
    double* f0hat = nullptr;  // dS o f0
    double* dgamma0 = nullptr;
    double gamma0 = 0.0;      // host copy of Gamma0
    int* sorder = nullptr;    // the 16 ns stencil entries e = 16 p + 4 b + a sorted by (grid node, e)
    int* snode = nullptr;     // their grid nodes in that order (both null when ns > SHEET_SORT_MAX)
    double* gj = nullptr;     // blocked Gauss-Jordan scratch: LU (32 x 32), Y, Z (32 x ns), L_R (ns x 32), perm, gperm
    double* work = nullptr;   // 12 ns doubles of solve scratch
    double* mwork = nullptr;  // several-body solve scratch (allocated by the first such solve)
    // surface pressure (pf_pressure_setup): unit normals (ns each), the face
    // stencils (per point 16 indices and weights: u lattice x, y then v lattice
    // x, y, 4 nodes each), the node stencils of C_s (ns x 64), and the factor of
    // the jump operator augmented with the gauge row (an (ns + 1) system)
    double* pnx = nullptr;
    double* pny = nullptr;
    int* fidx = nullptr;
    double* fwt = nullptr;
    int* ci = nullptr;
    int* cj = nullptr;
    double* cw = nullptr;
    struct pf_schur_s* jump = nullptr;
    int pbox[4] = {0, -1, 0, -1};   // cell-centre box (i0, i1, j0, j1) the surface faces can reach
    double* scal = nullptr;   // device scalars: s0, Gamma1, Gamma2, -, new-vortex x[2], y[2]
    int* rows = nullptr;      // lowest and highest grid row of the stencils (device): the rows psi is read at
    double* ewpart = nullptr; // surface sums: partial sums (ns x EW_SPLIT_MAX) and a done counter per point
    unsigned* ewdone = nullptr;
    double* gpart = nullptr;  // partial sums of Gamma (EW_SPLIT_MAX)
    double* sval = nullptr;   // R_s f dx^2 per sorted entry (16 ns; null as sorder)
};
constexpr int EW_SPLIT_MAX = 16;

// 1 / p within one unit in the last place of the division
// (tests/host/recip_check.cu): one step of the hyperpower (Schulz) iteration of order three,
// r (1 + e + e^2) with e = 1 - p r, from the hardware's 20-bit estimate r: e^3
// is about 2^-60, and one rounding; p normal and away from the ends of the
// range, else the division itself.  (Three dependent FP64 instructions of 64
// clocks; it stands in the serial chain of k_bgj_panel.)
__device__ __forceinline__ double fast_recip(double p) {
    const int ef = (__double2hiint(p) >> 20) & 0x7FF;
    if (ef < 64 || ef > 1982) return 1.0 / p;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(p));
    const double e = fma(-p, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

pf_status schur_create(pf_plan p, int ns, pf_schur* out);
void schur_free(pf_schur s);
pf_status schur_factor_device(pf_plan p, pf_schur s);
pf_status invert_schur_matrix(pf_plan p, pf_schur s);
// Several bodies (Sec. 2.7): validate a partition (and count its edges); the
// device-level solve of pf_sheet_solve_multi with new vortices at device
// (vx, vy) and, when gw_dev is not null, the bodies' gamma_w read from the
// device; *out_dev receives the device address of s0 (B values) then the new
// strengths (one per edge).
pf_status multibody_check(const pf_multibody& mb, int ns, int* n_edges_total);
constexpr int MAX_EDGES = 2 * PF_MAX_BODIES;

// edges releasing a vortex, and the placement rule's data
struct EdgeGeo {
    int n;
    double ex[MAX_EDGES], ey[MAX_EDGES];   // geometric edge points
    double nx[MAX_EDGES], ny[MAX_EDGES];   // unit normal facing the free stream
    double first_dist;                // 10 dt |U_inf|
    long long last[MAX_EDGES];
};

// Point vortices (device FP64 arrays of n, or *dn of them) of a sheet solve.
// pairs: E_s L^-1 R_v Gamma is summed from them (no field w is read).
struct VortexSource {
    const double* X = nullptr;
    const double* Y = nullptr;
    const double* G = nullptr;
    int64_t n = 0;
    const int64_t* dn = nullptr;
    int64_t cap = 0;           // the most n or *dn can be
    int pairs = 0;
    unsigned long long* oob = nullptr;   // with pairs: counts the vortices off the grid, as the R_v it replaces
};
// Steps take the vortex sum while ns x capacity is at most this.  The sum costs
// 0.19 us a thousand pairs; the field's right-hand side (R_v and the 64-bit
// streamfunction) 35 us and 20 more for every 2^20 nodes of the padded torus.
// A stage by field and by sum just below the line: 256^2 96 and 95.7 us, 512^2
// 114.3 and 112.1, 768 x 512 190.6 and 183.3, 1000^2 223 and 193; at 1.3 times
// it 98 and 109, 115.7 and 131.2, 191.8 and 209.8, 222.7 and 231.2 (mixed).  On
// larger grids the sum is the faster one at the line in either precision: 1024^2
// 241 and 198 (FP64 447 and 392), 1500 x 1024 386 and 302 (778 and 680), 2048 x
// 1800 749 and 512 (1582 and 1319), and by up to 18 % at 1.3 times the line still.
inline int64_t vortex_pairs_max(int P, int Q) { return 180000 + (int64_t)P * Q / 10; }
// (a rule on the state's capacity: a captured step takes the route of the step it stands for)
inline bool vortices_summed(pf_plan p, int ns, int64_t cap) {
    return p->rhs_route == PF_RHS_AUTO && (int64_t)ns * cap <= vortex_pairs_max(p->P, p->Q);
}

// E_s L^-1 R_v Gamma into s->ewpart (vortex_rhs_chunks partial sums a
// point), sums of Gamma into s->gpart (as many), E_s L^-1 d_j of ne released
// vortices into unit[j ns + p]; their positions are read from newx, newy, or
// written there by the placement rule.
int vortex_rhs_chunks(int ns, int64_t cap);
pf_status vortex_rhs(pf_plan p, pf_schur s, const VortexSource& vs, int ne, const EdgeGeo* place, double* newx, double* newy,
                     double* unit);                                                               // sheet.cu
pf_status sheet_solve_multi_device(pf_plan p, pf_schur s, const void* w, const pf_multibody& mb, int ne,
                                   double* vx, double* vy, double* f, const double* gw_dev,
                                   double** out_dev, const VortexSource* vs = nullptr);
// Generalized edge condition (Sec. 2.5) for the shedding mode: with on = 0 every
// edge sheds under the Kutta condition; otherwise edge e sheds only when its
// intermediate value lies outside [lo[e], hi[e]], and ends at the bound crossed.
struct EdgeBounds {
    int on = 0;
    double lo[2] = {0.0, 0.0};
    double hi[2] = {0.0, 0.0};
};
// vortices released by a solve: appended to a state's arrays at nv (dn[0] when use_dn)
struct Release {
    int n = 0;
    double *X = nullptr, *Y = nullptr, *G = nullptr;
    int64_t nv = 0, cap = 0;
    int64_t* dn = nullptr;
    int use_dn = 0;
    const double *newx = nullptr, *newy = nullptr;
    int* status = nullptr;
};
// bodies of at most this many points are solved by one cluster (k_sheet_small)
constexpr int SHEET_SMALL = 256;
struct SheetSmall {
    int mode, ns, nc, nedge, k1, k2;
    EdgeBounds eb;
    pf_motion m;
    double param_h;
    const double* param_d;
    const double* gpart;             // not null: param = gsign * sum gpart
    int ngpart;
    double gsign;
    const double *x, *y, *ds, *S, *Sinv, *f0, *f0hat, *gamma0;
    const double* part;              // E L^-1 w: `chunks` partial sums a point
    int chunks;
    const double* unit;
    double *f, *scal, *f0hat_out;
    Release rel;
    const int *sorder, *snode;       // sval (nullable): R_s f dx^2 at each node's first sorted entry
    const double *swx, *swy;
    double* sval;
};
pf_status sheet_small(pf_plan p, const SheetSmall& a);                                            // sheet.cu
pf_status sheet_f0_small(pf_plan p, pf_schur s);                                                  // sheet.cu

// What a time step adds to a sheet solve (all of it only while ns <=
// SHEET_SMALL, but for vs->pairs): the vortices the right-hand side or the
// total circulation comes from (param = gsign x sum Gamma), the placement of
// the released ones and their release, the sheet's node values.
struct SheetStep {
    const VortexSource* vs = nullptr;
    const EdgeGeo* place = nullptr;
    double gsign = 0.0;
    Release rel;
    bool nodes = false;
};
// param_dev (nullable): device copy of `param` read by the kernels instead
pf_status sheet_solve_device(pf_plan p, pf_schur s, const void* w, const pf_motion& m, int mode, double param,
                             const double* param_dev, int n_edges, const int* edges, double* vx, double* vy, double* f,
                             const EdgeBounds& eb = EdgeBounds(), const SheetStep& step = SheetStep());
// w += R_s f  (device f of ns doubles, w real[nx*ny])
pf_status sheet_deposit(pf_plan p, pf_schur s, const double* f, void* w);
// allocate what the sheet solves of steps of a state of this capacity allocate on first use
pf_status sheet_solve_reserve(pf_plan p, pf_schur s, int64_t cap);

// step.cu: asynchronous state transfers used by the request server
pf_status state_load_async(pf_state s, const double* X, const double* Y, const double* G, int64_t nv, double t);
pf_status state_store_async(pf_state s, double* X, double* Y, double* G, int64_t* nv);
int64_t state_capacity(pf_state s);
// One pf_step of (p, s, k) captured on the plan's stream and instantiated
// (the capture runs nothing; s's host counts are left as they were).  The
// body must be fixed in time; the factor at its pose and every buffer a step
// of the state's capacity uses are made ready first (this may synchronise the
// plan's stream).  released: the vortices one step appends.
pf_status step_graph_create(pf_plan p, pf_state s, const pf_body_kinematics& k, double dt, int scheme,
                            cudaGraphExec_t* out, int* released);
// the host counts after one launch of a captured step
void step_graph_advance(pf_state s, int released, double dt);
