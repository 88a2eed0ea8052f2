// Build-time generator of the FP32 predictor's reference-stiffness contractions (Sec. 4.3,
// Eq. ader4: R_{k,t} = sum_d S^_d (dt adj(J_k) F)_d; Eq. TAvectors: the volume term with
// S^_d transposed).
//
// The stiffness matrices S^_d[m][l] = int phi_m d/dxi_d phi_l of the reference tetrahedron are
// universal, so the contraction of one column b[(d, j)] (the 3 Np pre-contracted flux values of
// one sub-tet, variable and time slice) with them can be written out with the matrix entries
// as instruction immediates: every multiply-add reads its coefficient from the instruction
// stream (no shared-memory or constant-cache traffic for S^) and the entries that vanish are
// not multiplied at all.  The entries are those of build_ref() (the values the library uploads
// for its other kernels), rounded to FP32 as the FP32 form uses them.  Entries that vanish in
// exact arithmetic come out of build_ref()'s extended-precision solve at the 1e-19 level; those
// below 1e-13 of the largest entry are taken as the zeros they are.  The accumulation runs over
// (d, j) in increasing order for every m, as a dense loop would.
//
// Usage: gen_sref <output header>
#include <cmath>
#include <cstdio>
#include <string>
#include <vector>

#include "refelem.hpp"

namespace {

// Row stride (floats) of a column in shared memory: a multiple of 4 floats (16-byte rows for
// vector loads) with an odd number of 16-byte groups, so that the eight lanes of a quarter
// warp that load consecutive columns hit eight different bank groups.
int column_stride(int kk) {
  int g = (kk + 3) / 4;
  if (g % 2 == 0) ++g;
  return 4 * g;
}

std::string lit(float x) {
  char buf[64];
  std::snprintf(buf, sizeof buf, "%af", (double)x);
  return buf;
}

// acc[m] += sum_{kk < KK} C(m, kk) b[kk], kk = d Np + j, in increasing kk for every m.
template <typename Coef>
void emit_body(FILE* f, int np, Coef coef) {
  const int kk_n = 3 * np;
  const int groups = (kk_n + 3) / 4;
  for (int q = 0; q < groups; ++q) {
    std::fprintf(f, "    {\n      const float4 x = *reinterpret_cast<const float4*>(b + %d);\n", 4 * q);
    static const char* comp[4] = {"x.x", "x.y", "x.z", "x.w"};
    for (int i = 0; i < 4; ++i) {
      const int kk = 4 * q + i;
      if (kk >= kk_n) break;
      for (int m = 0; m < np; ++m) {
        const float c = coef(m, kk);
        if (c == 0.0f) continue;
        std::fprintf(f, "      acc[%d] = fmaf(%s, %s, acc[%d]);\n", m, lit(c).c_str(), comp[i], m);
      }
    }
    std::fprintf(f, "    }\n");
  }
}

// out[d Np + j] = sum_l D[d][j][l] x[l]: the reference gradient of a nodal polynomial.
void emit_gradient(FILE* f, const afe::RefData& r) {
  const int np = r.Np;
  double dmax = 0.0;
  for (int d = 0; d < 3; ++d)
    for (int j = 0; j < np; ++j)
      for (int l = 0; l < np; ++l) dmax = std::fmax(dmax, std::fabs(r.D[d][j][l]));
  std::fprintf(f,
               "  // out[d Np + j] = sum_l D[d][j][l] x[l]: reference gradient of a sub-tet polynomial\n"
               "  static __device__ __forceinline__ void gradient(const float (&x)[%d], float* out) {\n"
               "    float a[%d];\n",
               np, np);
  for (int d = 0; d < 3; ++d) {
    std::vector<bool> seen(np, false);
    for (int l = 0; l < np; ++l)
      for (int j = 0; j < np; ++j) {
        const double c = r.D[d][j][l];
        if (std::fabs(c) < 1e-13 * dmax) continue;
        if (seen[j]) std::fprintf(f, "    a[%d] = fmaf(%s, x[%d], a[%d]);\n", j, lit((float)c).c_str(), l, j);
        else std::fprintf(f, "    a[%d] = %s * x[%d];\n", j, lit((float)c).c_str(), l);
        seen[j] = true;
      }
    for (int j = 0; j < np; ++j) std::fprintf(f, "    out[%d] = %s;\n", d * np + j, seen[j] ? ("a[" + std::to_string(j) + "]").c_str() : "0.f");
  }
  std::fprintf(f, "  }\n");
}

// Entries of S^ that vanish in exact arithmetic are set to the zeros they are.
void drop_zeros(afe::RefData* r) {
  const int np = r->Np;
  double smax = 0.0;
  for (int d = 0; d < 3; ++d)
    for (int m = 0; m < np; ++m)
      for (int j = 0; j < np; ++j) smax = std::fmax(smax, std::fabs(r->S[d][m][j]));
  for (int d = 0; d < 3; ++d)
    for (int m = 0; m < np; ++m)
      for (int j = 0; j < np; ++j)
        if (std::fabs(r->S[d][m][j]) < 1e-13 * smax) r->S[d][m][j] = 0.0;
}

// The reference gradient (and S^ at N = 1) for the FP64 form: the entries sit in constant memory and reach the
// multiply-adds as constant operands (immediates hold 32 bits).
void emit_f64(FILE* f, const afe::RefData& r) {
  const int np = r.Np;
  double dmax = 0.0;
  for (int d = 0; d < 3; ++d)
    for (int j = 0; j < np; ++j)
      for (int l = 0; l < np; ++l) dmax = std::fmax(dmax, std::fabs(r.D[d][j][l]));
  // S^ itself at N = 1 only (above, the FP64 form's contraction runs on the tensor cores)
  std::string contract[2];
  for (int tr = 0; tr < 2 && r.N == 1; ++tr) {
    std::vector<double> k;
    char line[160];
    for (int kk = 0; kk < 3 * np; ++kk)
      for (int m = 0; m < np; ++m) {
        const double v = tr ? r.S[kk / np][kk % np][m] : r.S[kk / np][m][kk % np];
        if (v == 0.0) continue;
        std::snprintf(line, sizeof line, "    acc[%d] = fma(kStiffness%d[%d], b[%d], acc[%d]);\n", m, tr, (int)k.size(), kk, m);
        contract[tr] += line;
        k.push_back(v);
      }
    std::fprintf(f, "static __device__ __constant__ double kStiffness%d[%d] = {", tr, (int)k.size());
    for (size_t i = 0; i < k.size(); ++i) std::fprintf(f, "%s%a", i ? ", " : "", k[i]);
    std::fprintf(f, "};\n");
  }
  std::vector<double> c;
  std::string g;
  char buf[160];
  for (int d = 0; d < 3; ++d) {
    g += "    for (int j = 0; j < " + std::to_string(np) + "; ++j) a[j] = 0.0;\n";
    for (int l = 0; l < np; ++l)
      for (int j = 0; j < np; ++j) {
        if (std::fabs(r.D[d][j][l]) < 1e-13 * dmax) continue;
        std::snprintf(buf, sizeof buf, "    a[%d] = fma(kGradient%d[%d], x[%d], a[%d]);\n", j, r.N, (int)c.size(), l, j);
        g += buf;
        c.push_back(r.D[d][j][l]);
      }
    for (int j = 0; j < np; ++j) {
      std::snprintf(buf, sizeof buf, "    out[%d] = a[%d];\n", d * np + j, j);
      g += buf;
    }
  }
  std::fprintf(f, "static __device__ __constant__ double kGradient%d[%d] = {", r.N, (int)c.size());
  for (size_t i = 0; i < c.size(); ++i) std::fprintf(f, "%s%a", i ? ", " : "", c[i]);
  std::fprintf(f, "};\n");
  std::fprintf(f, "template <>\nstruct SrefFP64<%d> {\n", r.N);
  if (r.N == 1)
    for (int tr = 0; tr < 2; ++tr)
      std::fprintf(f, "  static __device__ __forceinline__ void %s(const double* b, double (&acc)[%d]) {\n%s  }\n",
                   tr ? "contract_t" : "contract", np, contract[tr].c_str());
  std::fprintf(f, "  static __device__ __forceinline__ void gradient(const double (&x)[%d], double* out) {\n    double a[%d];\n%s  }\n};\n\n", np, np, g.c_str());
}

}  // namespace

int main(int argc, char** argv) {
  if (argc != 2) {
    std::fprintf(stderr, "usage: %s <output header>\n", argv[0]);
    return 2;
  }
  FILE* f = std::fopen(argv[1], "w");
  if (!f) {
    std::perror(argv[1]);
    return 1;
  }
  std::fprintf(f,
               "// Generated at build time by gen_sref.cpp from build_ref(): the FP32 predictor's\n"
               "// reference-stiffness contractions with S^ as immediates.  Do not edit.\n"
               "#pragma once\n\nnamespace afe {\n\n"
               "template <int N>\nstruct SrefFP32;\n\n");
  // the FP64 gradients follow in a section of their own, for the translation units that ask
  for (int N = 1; N <= 3; ++N) {
    static afe::RefData r;
    if (!afe::build_ref(N, &r)) {
      std::fprintf(stderr, "build_ref(%d) failed\n", N);
      return 1;
    }
    const int np = r.Np, kk_n = 3 * np;
    drop_zeros(&r);
    int nz_p = 0, nz_v = 0;
    for (int d = 0; d < 3; ++d)
      for (int m = 0; m < np; ++m)
        for (int j = 0; j < np; ++j) {
          nz_p += (float)r.S[d][m][j] != 0.0f;
          nz_v += (float)r.S[d][j][m] != 0.0f;
        }
    std::fprintf(f, "// node order j = 0 .. Np-1 (barycentric multi-indices alpha_0 alpha_1 alpha_2 alpha_3):");
    for (int j = 0; j < np; ++j)
      std::fprintf(f, "%s %d%d%d%d", j % 10 == 0 ? "\n//" : "", r.alpha[j][0], r.alpha[j][1], r.alpha[j][2], r.alpha[j][3]);
    std::fprintf(f, "\ntemplate <>\nstruct SrefFP32<%d> {\n", N);
    std::fprintf(f, "  static constexpr int KK = %d;   // 3 Np pre-contracted values per column\n", kk_n);
    std::fprintf(f, "  static constexpr int KKS = %d;  // column stride in shared memory (floats)\n",
                 column_stride(kk_n));
    std::fprintf(f, "  static constexpr int kTerms = %d, kTermsT = %d;  // non-zero entries used\n", nz_p, nz_v);
    std::fprintf(f,
                 "  // acc[m] += sum_{d,j} S^_d[m][j] b[d Np + j]: the reference-stiffness contraction of\n"
                 "  // the predictor's right-hand side\n"
                 "  static __device__ __forceinline__ void contract(const float* __restrict__ b, float (&acc)[%d]) {\n",
                 np);
    emit_body(f, np, [&](int m, int kk) { return (float)r.S[kk / np][m][kk % np]; });
    std::fprintf(f, "  }\n");
    std::fprintf(f,
                 "  // acc[m] += sum_{d,j} S^_d[j][m] b[d Np + j]: the volume term's contraction\n"
                 "  static __device__ __forceinline__ void contract_t(const float* __restrict__ b, float (&acc)[%d]) {\n",
                 np);
    emit_body(f, np, [&](int m, int kk) { return (float)r.S[kk / np][kk % np][m]; });
    std::fprintf(f, "  }\n");
    emit_gradient(f, r);
    std::fprintf(f, "};\n\n");
  }
  std::fprintf(f, "#ifdef AFE_SREF_F64\ntemplate <int N>\nstruct SrefFP64;\n\n");
  for (int N = 1; N <= 3; ++N) {
    static afe::RefData r;
    if (!afe::build_ref(N, &r)) return 1;
    drop_zeros(&r);
    emit_f64(f, r);
  }
  std::fprintf(f, "#endif\n\n");
  std::fprintf(f, "}  // namespace afe\n");
  std::fclose(f);
  return 0;
}
