// Node-shared Krylov kernel: one real Lanczos sequence per node, in
// fixed-point arithmetic on the integer pipe, serves every pole of the node
// (md_krylov.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

#include "md_internal.h"
#include "md_solver.h"

namespace md {

constexpr int kKryMaxQ = 4;        // stencil half-widths 1..4 (fd_order <= 8)
constexpr int kKryMaxPoles = 64;
constexpr int kKryChunkRows = 32;  // projector rows of one atom a warp sums in one go
constexpr int kKryVec = 32;        // Krylov vectors kept between two updates of the solution vectors
constexpr int kKryMaxDepth = 40;   // planes of a CTA's slab (bounds the exact partial sums)

struct KrylovParams {
    // operator A = (H_R - shift) / scale, weights in two signed 31-bit limbs
    // (value = hi 2^-31 + lo 2^-62), wf the pair {(float)lo, (float)hi}; the
    // kernel with FP32 mixed terms takes wf, the exact one wl
    int n[3];
    int periodic[3];
    const double* V;
    double scale, shift;
    int wh[3][kKryMaxQ], wl[3][kKryMaxQ];
    unsigned long long wf[3][kKryMaxQ];
    // nonlocal projectors
    long long n_atoms;
    const int* proj_i0;
    const int* proj_len;
    const unsigned char* proj_rows;
    const int4* proj_fx;           // [atom][axis][kMaxProjWin] unit tables: g (hi, lo), d g (hi, lo), halved
    const double* proj_fxc;        // [atom][4] 64 E_l C_l^2 of the unit tables
    int rec_words;                 // 4 projector rows per word and region point
    int exact;                     // mixed terms of products: 64-bit integers, else FP32
    // FP64 operator of the final check of a mixed solve with FP32 mixed terms
    int check;
    double coef[3][kKryMaxQ];
    double dV, e_s, e_p;
    const int* pl_ptr;
    const int* pl_atom;
    const double2* pl_val64;
    // work: node list in scheduling order
    int n_work;
    const int* list;
    const NodeDesc* nodes;
    unsigned int* work_counter;
    unsigned long long timeout_ns;
    unsigned long long* t_start;   // when the call's first CTA ran (0: not yet), shared by its launches
    // per-CTA scratch layout
    char* scratch;
    size_t cta_bytes;
    size_t off_up, off_w, off_rec, off_rows, off_ktab, off_xtab, off_chunk, off_cpart;
    int row_cap;
    int win_x;                     // x window of the tables, points
    int smem_bytes;                // dynamic shared memory of the launch
    // poles (all solves but Lanczos rules)
    int P;
    const double2* z;
    double tol, tol_conv;          // of the true residual, and of the recurrence's
    int maxit;
    double2* x_src;                // [node * P + pole]
    int* status;
    int* iters;
    double* resid;
    int* n_rel;
    // Solution vectors: with vec, x_jp is accumulated over the region (in ckpt,
    // or in scratch) and used for the outputs below
    int vec;
    size_t off_x, off_p, off_hist, off_coef;
    double2* ckpt;                 // NULL or checkpoint base
    const long long* ckpt_off;     // point offset of system (node*P + pole) in ckpt
    double* fused_dLdV;            // fused adjoint, see SolveParams
    const double* fused_a;
    const double* fused_b;
    const double2* w;
    double* dm_rows;
    const long long* dm_off;
    // Lanczos rules: K > 0 stops after K steps and stores the coefficients
    int K;
    double breakdown_tol;
    double* alpha;                 // [node][K]
    double* beta;
    int* k_used;
    int* node_status;
};

// Shared memory of one CTA for a slab of `depth` planes of m0 x m1 points,
// without the nonlocal tables (which take what is left of the launch's
// dynamic shared memory).
size_t kry_u_bytes(int q, int m0, int m1, int depth);
size_t kry_static_smem_bytes(int nonlocal);
// Scratch of the solution vectors' coefficients, per CTA.
size_t kry_vec_bytes(int P);
int kry_max_threads();
// Resident clusters of csz CTAs; 0 if the shape cannot run.
int kry_max_clusters(int q, int nonlocal, int csz, int block, size_t smem);
cudaError_t launch_krylov(const KrylovParams& P, int q, int nonlocal, int csz, int grid, int block, size_t smem,
                          cudaStream_t stream);
// Unit projector tables and their coefficients; *bad is set if some atom's
// normalisation leaves the fixed-point range.
cudaError_t launch_proj_fixed(long long n_atoms, const int* len, const double* dtab, const double* gtab,
                              const double* C, double dV, double e_s, double e_p, int4* fx, double* fxc, int* bad,
                              cudaStream_t stream);

}  // namespace md
