// idugks_internal.h -- data shared by the host side (idugks_host.cpp) and the
// kernels (idugks_kernels.cu) of libidugks.  Not part of the C ABI.
#pragma once

#include <cstddef>
#include <cstdint>

namespace idg {

constexpr int kMaxVel = 16384;
constexpr int kMaxHist = 1 << 16;  // residual-history ring (iterations)
constexpr int kCellP = 16;         // per-cell / per-face coefficient records
constexpr int kRaw = 11;           // raw velocity moments kept per cell / face
constexpr int kSMs = 152;  // streaming multiprocessors of a GB300
constexpr int kNoAllocMaxCells = 16384;  // cell limit of idg_get_moments_noalloc

// Everything one kernel launch needs, passed by value.  Device pointers point
// into the caller's workspace.  "T" below is the storage precision (float for
// IDG_MIXED, double for IDG_FP64); "acc" entries are 8 bytes: a float-float
// pair (hi, lo) in mixed precision, a double in FP64.  Distributions are kept
// relative to one reference Maxwellian M_ref (f = M_ref + dev).
struct KParams {
    // sizes
    int N, Nv, nf, ni, nj, nvx, nvy;
    int K, shakhov, limiter;
    int per_i, per_j;
    // cells
    const double *area;    // [N]
    const double *dtimp;   // [N]
    const double *adt;     // [N] area / dtimp
    const int *cface;      // [N][4] faces in slots west, east, south, north
    const int *cnb;        // [N][4] neighbour across the slot (-1 ghost)
    const int *csign;      // [N][4] +1 if the cell is the L side of that face
    const void *crT;       // [N][8] T: face midpoint minus centroid, per slot
    const void *clsgT;     // [N][8] T: least-squares weight vector per slot
    const void *cnT;       // [N][4][2] T: outward normal per slot, sign*nx, sign*ny
    const void *cslotT;    // [N][4][2] T: sign*nx*S, sign*ny*S per slot (micro sweeps)
    const int *scode;      // [2][N][4] forward, backward: role of each slot's neighbour in that micro sweep
                           // (scheduled sweeps of an unstructured mesh; null on a structured block)
    void *sgeo;            // [2][N][8] T forward, backward: what the line sweeps read of a cell (k_sweep_lines);
                           // entry 6, the cell's diagonal base, is written every iteration (null if unstructured)
    // faces
    const int *fL, *fR;    // [nf]
    const double *fgeo;    // [nf][7] nx, ny, S, rLx, rLy, rRx, rRy
    const void *fgeoT;     // [nf][8] T copy of fgeo
    const int *fbc;        // [nf] -1 interior, else boundary kind
    const int *fside;      // [nf] boundary side or -1
    const double *bconst;  // [nf][2] boundary faces: sum_out w (xi.n_out) G_ref, sum_in w |xi.n_out| G_bnd
    // velocity tables
    const double *ux, *uy, *w;   // [Nv]
    const double *gref;          // [Nv] reduced reference Maxwellian G
    const float *uxf, *uyf, *wf, *greff;  // float copies
    const void *bdevG, *bdevH;   // [4][Nv] T: boundary Maxwellian minus M_ref (wall: unit density)
    // gas and numerics
    double dt, h, mu_ref, RT_ref, omega, Pr, gam, lusgs_omega;
    double venkat_k3;  // cube of the limiter's smoothing constant: eps^2 = venkat_k3 * area^(3/2)
    // reference Maxwellian parameters and its discrete moments
    double rho_r, U_r, V_r, RT_r;
    double iRT_r, iAref;     // 1 / RT_r, 2 RT_r / rho_r (one over rho_r lambda_r)
    double iRT_ref, iK2, pc0; // 1 / RT_ref, 1 / (K + 2), (1 - Pr) / (K + 4)
    double mref_raw[kRaw];     // raw moments: G: 1,x,y,xx,xy,yy,x|xi|^2,y|xi|^2; H: 1,x,y
    double mref_flux[4][2];    // sum w psi xi_a M_ref, psi = 1, xi_x, xi_y, energy
    // state and work (T2 = {G, H} deviation pairs of the storage type)
    void *f;        // [N][Nv] T2 state f~ - M_ref
    void *fbp;      // [N][Nv] T2 fb+ - M_ref
    void *F;        // [nf][Nv] T2 fb at the face (minus M_ref), then the flux of (f_face - M_ref)
    void *ftie;     // [nf][max(nvx, nvy)] T2 interior faces: fb from the R side at velocities along the face (tie_slot())
    void *dst;      // [N][Nv] T2 residual, Delta* then Delta (the memory of fbp)
    double *W;      // [N][4]
    void *cellraw;  // [N][kRaw] acc raw moments of f~ - M_ref
    void *cellA;    // [N][16] T: equilibrium at W^n (14), c1, c2 of fb+
    double *cellq;  // [N][2]  heat flux of f at cells (from f~^n)
    void *cellpT;   // [N][16] T: equilibrium at the predicted state (14), collision rate, micro diagonal base
    void *faceraw;  // [nf][12] acc raw moments of fb - M_ref, wall outgoing sum
    double *facerw; // [nf] wall density rho_w (1 elsewhere)
    void *faceA;    // [nf][16] T: face equilibrium (14), a, b of Eq. (18)
    void *phiraw;   // [nf][4] acc moments of the deviation flux
    double *phi;    // [nf][4]
    double *rw;     // [N][4]
    // macroscopic LU-SGS work (T = storage precision of the sweep)
    void *mrec;     // [N][24] T: R, 1/D, own base state, per slot (S/2) n_out, (omega/2) Lambda
    void *mline;    // [6][nslot][4] T: the record as k_macro_lines reads it (null if unstructured), cell slots by line_slot()
    void *mdW;      // [N][4] T increments (Delta W* then Delta W); k_macro_lines: [nslot][4]
    void *mdW2;     // [N][4] T second increment buffer of the point relaxation (else null)
    double *mpart;  // [ceil(N/32)] block partial sums of ||R/Omega||^2
    double *res;    // [kMaxHist] absolute residual per iteration
    int *iter;      // [1] device iteration counter
    int *status;    // [1] device status word
    // launch shape of the wavefront kernels: velocities per CTA and cell
    // slots of the micro sweeps, prefetch depths asked for (steps; 2, 4 or 8)
    int sweep_tv, sweep_pc, sweep_stages, macro_stages;
    int row_warps;   // warps per cell of k_cell_moments (1, 2, 4)
    int cpb;         // cells per block of the per-(cell, velocity) kernels
    int sweep_tuned; // set by the caller: 1 sweep_tv, 2 sweep_vpt, 4 sweep_stages
    // the tile that runs (sweep_shape()): threads per cell of a block and
    // velocities per thread; line sweeps: sweep_g of those threads neighbours in
    // one warp, entries of a border ring
    int sweep_ktv, sweep_kvpt, sweep_g, sweep_ring;
    int wait_polls;  // polls after the first before a wait between warps gives up (idg_set_wait_limit)
    int sweep_vpt;  // consecutive velocities per thread in the micro sweeps (1, 2, 4)
    int macro_kind; // macroscopic LU-SGS on a structured block: 0 hyperplane slots (k_macro_sweep),
                    // 1 one thread per line of cells (k_macro_lines)
    int relax_sweeps;  // macroscopic predictor: 0 LU-SGS, n >= 1 n point-relaxation sweeps
    // unstructured meshes: the sweeps' schedule (null on a structured block,
    // whose sweeps walk the i+j hyperplanes): sched [2][N] cells in processing
    // order for the forward then the backward sweep, sptr the step offsets
    // into each ([nsteps_f + 1] then [nsteps_b + 1]); the cells of one step
    // depend on none of each other
    const int *sched, *sptr;
    const int *snb;  // [2][N][4] in the order of sched: the cell's neighbours already swept, by slot (else -1)
    int nsteps_f, nsteps_b;
    // linearised diffuse wall of the micro sweeps (Eq. 33-35), implicit_wall
    // = 1: per face, wallS the inner cell's outgoing sum sum_out w (xi.n_out)
    // G~ of the last iteration, walldrg the ghost density increment drho_g
    // (wall faces only; else null); wallok 0 after a restart (no last
    // increment), 1 once an iteration has stored wallS
    int implicit_wall;
    double *wallS, *walldrg;
    int *wallok;
};

// kernels of one iteration, in launch order
enum KType {
    KT_CELL_MOM, KT_CELL_PAR, KT_FBP, KT_FACE_MOM, KT_FACE_PAR, KT_FACE_FLUX, KT_FACE_PHI,
    KT_MACRO_PRE, KT_MACRO_SWEEP, KT_MACRO_POST, KT_MICRO_RES, KT_SWEEP, KT_COUNT
};

// How one iteration is launched over one or many instances: the instances'
// parameters in device memory, per-kernel prefix sums of blocks per instance
// (null for a single instance), activity flags (null: all active), and the
// block shapes common to all instances.
struct Plan {
    const KParams *hparams;  // a single instance: its parameters on the host, passed by value; null for a batch
    const KParams *dparams;
    const int *doff;     // [KT_COUNT][ninst + 1]
    const int *dactive;  // [ninst]
    int ninst;
    int nblocks[KT_COUNT];
    int macro_threads, sweep_threads;
    size_t macro_smem, fwd_smem, bwd_smem;
    int macro_stages, sweep_stages, limiter_any, sweep_vpt;
    int macro_kind;      // KParams::macro_kind of every instance
    int any_seam;        // 1: an instance has a periodic direction (k_macro_lines' seam terms)
    int explicit_dugks;  // 1: launch_iteration runs one explicit DUGKS step (Eq. 21)
    int relax_sweeps;    // macroscopic predictor of every instance (KParams::relax_sweeps)
    int sched;           // 1: the instances are unstructured (scheduled sweeps)
    size_t sched_smem;   // shared memory of the scheduled macroscopic sweep (0: increments in global memory)
};

// launch shape of the micro sweeps: KParams::sweep_ktv, sweep_kvpt, sweep_g,
// sweep_ring, what the caller set and the rest by size; vpt > 0 fixes the
// velocities per thread (one value for all instances of a batch)
void sweep_shape(KParams &p, bool fp64, int vpt = 0);
// whether shared memory holds what the caller asks of the micro sweeps: sweep_tv,
// sweep_vpt and sweep_stages
bool sweep_request_fits(const KParams &p, bool fp64);

// kernel launchers (idugks_kernels.cu)
int configure_kernels(bool fp64);
int configure_sweeps(const Plan &plan, bool fp64);  // before a plan's first launch
void blocks_per_instance(const KParams &p, int out[KT_COUNT]);
int plan_shapes(const KParams *hp, int n, bool fp64, Plan &plan);
constexpr int kProfiled = 6;  // timed groups in launch_iteration(events)
int launch_iteration(const Plan &plan, bool fp64, void *stream, void **events = nullptr);
int launch_cell_moments(const KParams &p, bool fp64, double *out6_dev, void *stream);
// explicit DUGKS: W and the raw moments of the current f~ before the first step
int launch_explicit_prologue(const Plan &plan, bool fp64, void *stream);
// idg_get_moments_noalloc: raw moments in a static device array (no workspace)
int launch_cell_moments_noalloc(const KParams &p, bool fp64, int device, double *out6_dev, void *stream);
// absolute float64 G, H of [N][nvu] (the first nvu stored velocities of each
// cell) to / from the storage; to_dev sets the ghost velocities beyond nvu to M_ref
// float64 (G, H) [N][nvu] <-> the storage; deviation: the arrays hold f~ - M_ref
int launch_to_dev(const KParams &p, bool fp64, const double *G, const double *H, int nvu, void *stream,
                  bool deviation = false);
int launch_from_dev(const KParams &p, bool fp64, double *G, double *H, int nvu, void *stream,
                    bool deviation = false);

}  // namespace idg
