// FP64 complex products on the 5th-generation tensor cores by an exact split of the operands
// into bf16 digits; see tc_gemm64.cu.
#pragma once

#include "common.cuh"

// Most terms K of a product (2 K digit products stay below 2^23, for which the accumulators are joined).
constexpr int SG_KMAX = 248;
constexpr int SG_SLICES = 7;

// Split form of one R x K complex operand (K contiguous terms per row): bytes of the digits with
// `planes` planes (3: usable as the left or the right operand, 2: right operand only) and number
// of words for the row exponents and a mark for each group of eight rows.
size_t sg_form_bytes(int rows, int K, int planes);
inline int sg_form_exps(int rows) { return (int)ceil_div(rows, 8) * 9; }

// Split `batch` operands: row r, term k of operand z is src[z][r][k] (trans == false) or
// src[z][k][r] (trans), row-major with leading dimension ld and `stride` complex elements between
// the operands; src is complex64 (f32) or complex128.  Operands whose skip[z] != 0 are left out.
// digits: the highest of the seven digits that are written (five serve SG_HALF).
cudaError_t launch_sg_split(const void* src, bool f32, int64_t ld, int64_t stride, bool trans,
                            int rows, int K, int planes, int batch, unsigned char* form,
                            int32_t* exps, const int32_t* skip, cudaStream_t s, int digits = SG_SLICES);

// One term of a product set: output z (zlo <= z < zhi) adds A[z + zA] B[z + zB]^T of the split
// forms (members contiguous).
struct SgSeg {
  const unsigned char* A;
  const int32_t* eA;
  const unsigned char* B;
  const int32_t* eB;
  int planesA, planesB;
  int zA, zB, zlo, zhi;
};

// C[z] = C0[z] +- sum_g A_g B_g^T  (M x N outputs, K terms; neg: minus; C0 null: nothing added;
// C may be C0).  Every output takes part in at least one segment.  identity: C0 is the identity
// matrix.  C32 in the place of C: outputs rounded to complex64 (one segment, C0 null).
// maxabs[z] (or null): atomicMax of the bits of the largest |re|, |im| of output z as a
// float (rounded up by less than 2^-20; infinity for anything not finite).
// Products with skip[z] != 0 (or null) are left out, C[z] untouched; *any == 0 (or null) says that
// all of a one-job launch are.
struct SgJob {
  int nseg;
  SgSeg seg[2];
  bool neg, identity;
  const double2* C0;
  int64_t ldc0, sC0;
  double2* C;
  float2* C32;
  int64_t ldc, sC;
  int batch;
  uint32_t* maxabs;
  const int32_t* skip;
  const int32_t* any;
};

// Digit pairs kept: SG_FULL the 34 that count in FP64 (error about 2^-55 of the product of the
// row's and the column's largest entries, for digits of mixed sign; entries below 2^-56 of their row's
// largest count as zero, and so do subnormals), SG_HALF the fifteen of weights down to 2^-32 (error
// about 2^-36 of it: for corrections, and for residuals that are formed again), SG_SMALL the ten
// down to 2^-24 (2^-28).  They read seven, five and four digits.
enum SgDigits { SG_FULL, SG_HALF, SG_SMALL };

// One launch over one or two jobs of the same M, N, K (K <= SG_KMAX).  A wait that expires is
// recorded as DEV_TIMEOUT in *status.
cudaError_t launch_sg_gemm(int M, int N, int K, int njob, const SgJob* jobs, SgDigits digits,
                           int32_t* status,
                           long long wait_limit, cudaStream_t s);
