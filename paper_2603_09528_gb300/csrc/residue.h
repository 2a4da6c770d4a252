// Residue number systems of the float64 transform GEMMs (residue.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace tpt {

constexpr int kMaxModuli = 18;
constexpr int kMatrixBits = 54;       // transform-matrix rows: |X| <= 2^54
constexpr int kDataBits = 53;         // lines of the field: at least 53 bits of the line's maximum
constexpr int kMaxDataBits = 57;      // (14-bit digits, the top one of 15 bits and a sign)
constexpr int kResidueMaxK = 2048;    // contraction length (shared-memory tile of the y slicing)
constexpr int kOzakiMaxK = 576;       // contraction length a TPT_PREC_FP64_OZAKI plan accepts
// Residues of one pass of a transform; larger fields go in passes of whole z
// planes, so that a plan's workspace grows by at most this (16.7 M points of
// K = 512 lines, which is still 6.7 waves of GEMM tiles).
constexpr size_t kResidueScratch = size_t(512) << 20;

// The moduli for contraction length K: products and sums exact in float32.
struct ResidueSystem {
  int nm = 0, bits = 0, L = 0;        // moduli, bits of a line, bit length of P = prod p
  int p[kMaxModuli] = {};
  int y[kMaxModuli] = {};             // (P / p_i)^-1 mod p_i
  unsigned long long scale = 0;       // P / 2^L as a 64-bit binary fraction
};
bool residue_system(int K, ResidueSystem* s);

struct ResidueDir {                   // one direction of a plan
  bool ready = false;
  ResidueSystem sys;
  int kp = 0;                         // contraction length padded to 64
  void* tab[2] = {nullptr, nullptr};  // residues of Q^-1 (forward) and Q (inverse): rows of nm * kp bf16
  int* expo[2] = {nullptr, nullptr};  // their row exponents
};

constexpr int kMaxUp = 15;            // largest power of two a line is scaled up by
struct SliceConst {
  int nm, bits, L;
  float inv[kMaxModuli], p[kMaxModuli];
  float4 c[kMaxUp + 1][kMaxModuli];   // 2^(k + 14 j) mod p, centred, j = 0..3
};
struct MatrixConst {
  int nm;
  unsigned long long scale;
  int p[kMaxModuli], y[kMaxModuli];
};
struct ResiduePair {                  // two moduli folded together in the epilogue
  float inv1, p1, inv2, p2, f1, f2, e;
  int clo, chi;
};
struct ResidueGemm {
  int M, N, K, Kp, nm, npair, rm, n_fastest, accumulate, shift;
  long long sm, sn, f0;
  const int* expA;                    // row exponents of the two operands
  const int* expB;
  double* out;
  int* err;
  ResiduePair pair[(kMaxModuli + 1) / 2];
};

}  // namespace tpt
