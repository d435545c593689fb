// dispatch.h -- host-side launch descriptors and the per-(lattice, storage)
// operation tables that each translation unit exports.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "collide_v.cuh"

namespace lbm {

struct GeoH {
  int nx, ny, nz;
  int pitch;
  long long plane;
  int per[3];
};

struct Variant {
  int kind;    // 0: register kernel (one warp row per block row), 1: bulk-copy pipelined kernel,
               // 2: two steps per launch (pair_tma.cuh), X the widest strip
  int nv;      // kind 0: nodes per thread along x; kind 1: 4 for four nodes per consumer
               // thread (16-bit storage, A/B), else 0
  int bx;      // kind 0: threads per block along x (multiple of 32); kind 1: at most this
               // many resident blocks per SM (0: as many as fit)
  int by;      // kind 0: rows per block; kind 1: 1 for the staged bulk stores (A/B)
  int X;       // kind 1: tile width (nodes)
  int stages;  // kind 1: shared-memory ring depth
};

// Open boundaries of the square-cylinder benchmark (D2Q9, A/B, x non-periodic):
// a wall moving with (u_in, 0) half a spacing left of x = 0, and a Zou-He
// constant-density outlet (rho_out) at x = nx - 1.
// `fix` (step launches): apply the boundary rules to the gathered state; off
// for the first step after the state was written directly (lbm_init_equilibrium,
// lbm_set_populations), which holds f(t) as given, not a streamed state.
// For the helper kernels `on` already carries that condition.
struct OpenBC {
  int on, fix;
  double u_in, rho_out;
};

struct StepLaunch {
  OpenBC open;
  GeoH g;
  int collision;  // 0 TRT, 1 TRT-RLB, 2 P-TRT (BGK / RLB mapped by the caller)
  bool force;     // any force component non-zero
  CoefV<double> c;
  int* err;       // bounded-wait error word
  long long wait_ns;  // limit of each bounded wait (pipelined kernel)
  int extra_tx;       // test hook: bytes a stage waits for that never arrive
  int sms;        // multiprocessors of the device
  const void* src;
  void* dst;
  const uint8_t* mask;
  unsigned int* flag;
  unsigned int step;
  int layout;     // 0 A/B, 1 AA
  int parity;     // AA: 0 even (local) step, 1 odd (neighbour) step
  Variant v;
  // forcing: 1 Guo (Eq. source_guo), 2 simplified projection + G_i (Eq. source_simple,
  // Eq. Gi; two launches, phi = [D][N] values of the arithmetic precision)
  int scheme;
  void* phi;
  cudaStream_t stream;
};

struct AuxLaunch {
  OpenBC open;
  GeoH g;
  double rho0, F[3];
  void* pop;            // buffer holding the current state
  const uint8_t* mask;
  int layout;
  int parity;           // AA: parity of the number of completed steps
  cudaStream_t stream;
};

// Per-lattice descriptor and tile of the persistent batched kernel.
struct BatchDesc {
  GeoH g;
  CoefV<double> cd;
  CoefV<float> cf;
  long long off;  // byte offset of the lattice in each population arena
  int ntx;        // pipelined kernel: tiles per row at the variant's tile width
  int tile0;      // pipelined kernel: index of the lattice's first tile
};
struct BatchTile {
  int lat, x0, y0, z;
};
struct BatchLaunch {
  const BatchDesc* desc;
  const BatchTile* tiles;
  int ntiles;
  char* A;
  char* B;
  int nsteps;
  int parity0;          // 0: state in A, 1: state in B
  unsigned int step0;   // index of the first step (divergence records)
  unsigned int* flags;  // per-lattice divergence flags
  void* bar;            // BarrierWords
  unsigned int expected;
  long long timeout_ns;
  int collision;
  int bx, by, blocks;
  // pipelined variant (kind 1): tile width, ring depth, lattices, any force
  int kind, X, stages, nlat;
  bool force;
  cudaStream_t stream;
};

struct Ops {
  int Q, D, esize;
  // vector widths this storage supports for the fused kernel
  int nvs[4];
  int n_nv;
  cudaError_t (*step)(const StepLaunch&);
  cudaError_t (*init_eq)(const AuxLaunch&, const double* rho, const double* u);
  cudaError_t (*set_pop)(const AuxLaunch&, const double* f);
  cudaError_t (*get_pop)(const AuxLaunch&, double* f);
  cudaError_t (*macros)(const AuxLaunch&, double* rho, double* u);
  // FP64 diagnostics of the current state: u staged in `fields` in the arithmetic
  // precision (components 1 .. D of (1 + D) * N values), block partials [blocks][8]
  // (blocks <= rows), the eight sums in out[8] (mass, momentum, kinetic energy,
  // enstrophy, flag, 0)
  cudaError_t (*diag)(const AuxLaunch&, void* fields, double* partials, int blocks, double* out);
  // force on the solid nodes by momentum exchange (sum over fluid-to-solid links
  // of 2 e_i f*_i), partials [blocks][8] (slots 0..2), out[8] (slots 0..2)
  cudaError_t (*momentum)(const AuxLaunch&, int collision, const CoefV<double>& c, double* partials,
                          int blocks, double* out);
  // persistent batched kernel (cooperative launch) and its occupancy
  cudaError_t (*batch)(const BatchLaunch&);
  int (*batch_blocks_per_sm)(int collision, int threads);
  // pipelined persistent batched kernel (FP32 arithmetic storages only; else null)
  cudaError_t (*batch_tma)(const BatchLaunch&);
  int (*batch_tma_blocks_per_sm)(int collision, bool force, int X, int stages);
  // shared-memory bytes of the pipelined kernel for a tile width and ring depth (0: unsupported)
  size_t (*tma_smem)(int X, int stages);
  int mask_tile;  // its tile width on lattices with a solid mask (A/B)
  // the same for the kernel that takes two steps per launch (strip width, ring depth)
  size_t (*pair_smem)(int X, int stages);
};

// Strips of the kernel that takes two steps per launch: their width (a multiple
// of 64, at most X) and number for rows of nx nodes.  The last strip may be narrower,
// but not below 16 nodes, so that its neighbour's window does not reach
// past the row's end.  false: no such width (or a row below 32 bytes).
inline bool pair_strips(int nx, int esize, int X, int* sw, int* nstrips) {
  if (nx < 32 / esize) return false;
  const int n = (nx + X - 1) / X;
  for (int w = ((nx + n - 1) / n + 63) / 64 * 64; w >= 64; w -= 64) {
    const int k = (nx + w - 1) / w;
    if (k > 1 && nx - (k - 1) * w < 16) continue;
    *sw = w;
    *nstrips = k;
    return true;
  }
  return false;
}

// Staging buffers of the pipelined AA kernel's odd step: two on D2Q9 (its
// short collision would otherwise wait for the store warp), one on the 3-D
// lattices (whose staging rows are large).
inline constexpr int aa_odd_buffers(int Q) { return Q == 9 ? 2 : 1; }

// Shared memory the odd step of the pipelined AA kernel needs beyond its ring:
// the mbarriers (padded to 128 bytes) and aa_odd_buffers staging buffers of one
// row per plane of X + 2 * (16 / esize) elements, each rounded to 128 bytes;
// plus 128 bytes of alignment slack for where the ring ends.
inline constexpr size_t aa_odd_smem(int Q, int esize, int X) {
  return 128 + 128 +
         (size_t)aa_odd_buffers(Q) *
             (((size_t)Q * (size_t)(X + 2 * (16 / esize)) * (size_t)esize + 127) / 128 * 128);
}

// Shared memory the staged bulk stores of the pipelined A/B kernel (MODE 3)
// need beyond its ring: 128 bytes of alignment slack, four mbarriers (padded to
// 128 bytes) and two staging buffers of Q rows of X elements, each rounded to
// 128 bytes.
inline constexpr size_t tma_bs_smem(int Q, int esize, int X) {
  return 128 + 128 + 2 * (((size_t)Q * (size_t)X * (size_t)esize + 127) / 128 * 128);
}

// Per-direction collision constants from the rates and the force (host, FP64).
template <class L>
inline void fill_coef(double rho0, double wp, double wm_run, int collision, const double F[3],
                      CoefV<double>* c) {
  *c = CoefV<double>{};
  c->rho0 = rho0;
  c->cp = 1.0 - wp;
  c->cm = 1.0 - wm_run;
  const double hg = 1.0 - 0.5 * wp;
  for (int a = 0; a < 3; ++a) {
    c->Fh[a] = 0.5 * F[a];
    c->F[a] = F[a];
  }
  for (int i = 0; i < L::Q; ++i) {
    const double eF = L::cx(i) * F[0] + L::cy(i) * F[1] + L::cz(i) * F[2];
    const double w = L::w(i);
    c->fe[i] = 9.0 * w * eF * hg;
    c->fu[i] = -3.0 * w * hg;
    c->fa[i] = collision == 1 ? 1.5 * w * eF : 1.5 * w * eF * (2.0 - wm_run);
  }
  const double wd = L::w(L::Q - 1);  // diagonal weight of D2Q9 and D3Q19
  c->wp = wp;
  c->cpt = -c->cp / 3.0;
  c->cp2 = 0.5 * c->cp;
  c->cp4 = 0.25 * c->cp;
  // The moment-space form multiplies the momentum by cm + 36 wmd at every step
  // (wd = 1/36, sum over i of w_i e_ia^2 = 12 wd), so a rounding of either
  // constant compounds, by up to w- times 1e-16 a step.  From w- = 0.1 on, w- is
  // taken to the nearest value (within 5e-16) for which cm = 1 - 36 wmd is
  // exact.  Below, where that shift of w- would be the larger error, cm is 1 - w-
  // rounded (within 5.5e-17) and wmd is (1 - cm) / 36.  Relative velocity error
  // after 200 steps of a D2Q9 32^2 vortex at nu = 1 against an evaluation in long
  // double, pair by pair / grid / rounded cm: w- = 0.01 1.3e-15 / 8.9e-15 /
  // 1.3e-15, 0.03 3.9e-16 / 1.1e-15 / 3.4e-16, 0.1 1.1e-15 / 1.4e-16 / 8.8e-16,
  // 1.6 1.4e-14 / 3.0e-16 / 1.7e-14.  At nu = 0.01 the grid is the better one
  // from 0.02 (D2Q9) and 0.07 (D3Q19) on.
  const bool grid = wm_run >= 0.1;
  c->wmd = grid ? ldexp(nearbyint(ldexp(wm_run * wd, 55)), -55) : (1.0 - (1.0 - wm_run)) / 36.0;
  const double cmx = grid ? fma(-36.0, c->wmd, 1.0) : 1.0 - wm_run;
  c->cm2 = 0.5 * cmx;
  c->cm4 = 0.25 * cmx;
  for (int a = 0; a < 3; ++a) {
    c->hF[a] = hg * F[a];
    c->hF2[a] = 2.0 * hg * F[a];
    // F_i/2 (2 - w-) with the w- that cm stands for
    c->fax[a] = 1.5 * L::w(1) * F[a] * (1.0 + cmx);
    c->fad[a] = 1.5 * wd * F[a] * (1.0 + cmx);
  }
}

// The coefficients of forcing Scheme II: the F_i projection alone, without the
// symmetric Guo terms.
inline CoefV<double> coef_projection(CoefV<double> c) {
  for (int i = 0; i < kQMax; ++i) c.fe[i] = c.fu[i] = 0.0;
  for (int a = 0; a < 3; ++a) c.hF[a] = c.hF2[a] = 0.0;
  return c;
}

template <typename R>
inline CoefV<R> coef_cast(const CoefV<double>& d) {
  CoefV<R> c;
  c.rho0 = R(d.rho0);
  c.cp = R(d.cp);
  c.cm = R(d.cm);
  for (int a = 0; a < 3; ++a) {
    c.Fh[a] = R(d.Fh[a]);
    c.F[a] = R(d.F[a]);
  }
  for (int i = 0; i < kQMax; ++i) {
    c.fe[i] = R(d.fe[i]);
    c.fu[i] = R(d.fu[i]);
    c.fa[i] = R(d.fa[i]);
  }
  c.wp = R(d.wp);
  c.cpt = R(d.cpt);
  c.cp2 = R(d.cp2);
  c.cp4 = R(d.cp4);
  c.cm2 = R(d.cm2);
  c.cm4 = R(d.cm4);
  c.wmd = R(d.wmd);
  for (int a = 0; a < 3; ++a) {
    c.hF[a] = R(d.hF[a]);
    c.hF2[a] = R(d.hF2[a]);
    c.fax[a] = R(d.fax[a]);
    c.fad[a] = R(d.fad[a]);
  }
  return c;
}

const Ops* ops_d2q9_f64();
const Ops* ops_d2q9_f32();
const Ops* ops_d2q9_f16();
const Ops* ops_d2q9_bf16();
const Ops* ops_d3q19_f64();
const Ops* ops_d3q19_f32();
const Ops* ops_d3q19_f16();
const Ops* ops_d3q19_bf16();
const Ops* ops_d3q27_f64();
const Ops* ops_d3q27_f32();
const Ops* ops_d3q27_f16();
const Ops* ops_d3q27_bf16();

// Generic FP64 reductions over macroscopic fields (diag.cu).
struct DiagLaunch {
  GeoH g;
  int D;
  const double* rho;   // [N]
  const double* u;     // [D][N]
  const double* uref;  // [D][N] for the L2 error, else null
  const uint8_t* mask;
  double* partials;    // [blocks][8]
  double* out;         // [8]
  int blocks;
  cudaStream_t stream;
};
// out[k] = sum over blocks of partials[b][k] in block order (slot 6: maximum).
cudaError_t reduce_partials(const double* partials, int blocks, double* out, cudaStream_t st);
cudaError_t diag_l2(const DiagLaunch&);
cudaError_t copy_ceiling(const void* src, void* dst, size_t bytes, cudaStream_t st);

}  // namespace lbm
