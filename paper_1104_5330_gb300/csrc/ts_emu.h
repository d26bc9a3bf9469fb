// Host side of the double-precision passes on the tensor cores (ts_emu.cuh): the
// digit tables of the derivative matrices and the tile geometries of a grid.
#pragma once

#include "ts_internal.h"

namespace ts {

// One derivative matrix as the tensor cores' B operand: every row scaled by its own
// power of two (D = Dfix 2^-s), Dfix in eight balanced base-256 digits, the digits
// as f16 integers. Device layout, in 16-byte core columns of 8 K elements x `rows`
// matrix rows: [bias core][extra core, if any][kc K cores]; row j n + out of a K
// core is digit j of output `out` (n: outputs padded to a multiple of 8).
struct EmuMat {
  const uint16_t* dev = nullptr;
  const int* se = nullptr;   // 3 - s of every output (device)
  int nout = 0, n = 0, kc = 0, rows = 0, s = 0;   // s: the scale of a matrix whose rows share it
  int bytes() const { return (1 + kc + extra) * rows * 16; }
  int extra = 0;             // 1: the bias MMA's second core holds a leftover K element's digits
};

// Geometry of a pass that contracts two axes of a tile of Na x Nb x xw points.
struct EmuGeo {
  int xw, seq;               // 8 or 4; 1: the two digit copies share their memory
  int Na, Nb, hb;            // DFS axis, Fourier axis, half of the latter
  int ka, kb;                // K cores of 8 along a and b
  int nf, nz;                // functionals of the Fourier operand; nz of them in zero rows
  int sb1, d1, sb2, d2;      // bytes: row group and digit strides of the two digit copies
  int n1, n2, r1, r2, kc1, kc2;
  int mt1, mt2;              // 128-row tiles of the two contractions
  int exP;                   // pitch (doubles) of the exchange array
  int cols, dual, half;      // tensor-memory columns, two regions in flight, their distance
  int oC1, oC2, oB1, oB2, oCA, oEx, oMs, oLn, bytes;
  int threads;
};

constexpr int kEmuRadUnits = 3;   // (node, 8 columns) units of a tile that a thread holds

struct EmuRadGeo {
  int Nr, kc, left;          // K cores; 1: node N_r - 1 rides in the bias MMA
  int sb, d;                 // row group and digit strides of the digits
  int ng, go;                // output groups and outputs per group
  int n, rows;
  int cols, dual, half;
  int nb;                    // matrix buffers: ng, or 2 that the groups' matrices stream through
  int oA, oB, bB, oCA, oMs, bytes;   // bB: bytes of one group's matrix
  int threads;
};

constexpr int kEmuForms = 3;   // isotropic, linear and quadratic kernels (KF_*): their
constexpr int emu_functionals(int kf) { return kf == 0 ? 1 : kf == 1 ? 3 : 5; }   // Phi sums,
constexpr int emu_moments(int kf) { return kf == 0 ? 1 : kf == 1 ? 4 : 9; }       // moments,
constexpr int emu_weights(int kf) { return kf == 0 ? 1 : 3; }                     // Theta weights

struct EmuPlan {
  void* mem = nullptr;       // every table of the plan
  bool ang = false, plane = false, rad = false;      // which passes it covers,
  bool adj = false, planeT = false, radT = false;    // and which transposed ones
  EmuMat angD, angF[kEmuForms], plD, plF;
  EmuGeo gAng[kEmuForms], gPl;
  EmuMat adjD, adjF[kEmuForms], plTD, plTF;   // transposed operators
  EmuGeo gAdj[kEmuForms];
  EmuMat radM[8], radTM[8];  // one per output group
  EmuRadGeo gRad;
};

// Builds the plan of a grid (nullptr on failure or if no pass has one).
EmuPlan* emu_create(const ts_grid_desc& g, cudaError_t* e);
void emu_destroy(EmuPlan* p);

// Whether the plan covers a pass of a problem of these sizes: its tile numbers are
// decoded, and its offsets within a group formed, in 32 bits.
inline bool emu_small(const Dims& d) {
  return d.total < (1LL << 36) && d.nblk < (1LL << 31) && d.S_g < (1LL << 32);
}
inline bool emu_has_angular(const EmuPlan& e, const Dims& d) { return e.ang && emu_small(d); }
inline bool emu_has_plane(const EmuPlan& e, const Dims& d) { return e.plane && emu_small(d); }
inline bool emu_has_radial(const EmuPlan& e, const Dims& d) { return e.rad && emu_small(d); }

inline bool emu_has_angular_T(const EmuPlan& e, const Dims& d) { return e.adj && emu_small(d); }
inline bool emu_has_plane_T(const EmuPlan& e, const Dims& d) { return e.planeT && emu_small(d); }
inline bool emu_has_radial_T(const EmuPlan& e, const Dims& d) { return e.radT && emu_small(d); }

cudaError_t emu_angular(const EmuPlan& e, const Problem& p, const Tables<double>& t, bool cons,
                        const double* U, double* K, double sgn, bool collision, cudaStream_t s);
cudaError_t emu_plane(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                      const double* U, double* K, double sgn, cudaStream_t s);
cudaError_t emu_radial(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                       const double* U, const double* K, double sgn, bool tau, int mode, double* F,
                       double* Acc, double* Uout, double* out, double dt, cudaStream_t s);
// The transposed passes (see Launch::radial_T, plane_T, angular_T).
cudaError_t emu_radial_T(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                         const double* X, double scale, bool tau, double* lt, double* Ubar,
                         cudaStream_t s);
cudaError_t emu_plane_T(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                        const double* lt, double* Ubar, cudaStream_t s);
cudaError_t emu_angular_T(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                          const double* lt, const double* Ubar, const double* Us, double* gk,
                          double* ge, const double* lam, const double* lam_in, double* lam_out,
                          double* Kbar, double wl, double wu, cudaStream_t s);

}  // namespace ts
