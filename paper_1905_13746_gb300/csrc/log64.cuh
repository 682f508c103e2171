// FP64 natural logarithm of a positive number, for the fits' tables.
//
// FP64 runs at about two lanes per clock and SM on this part and CUDA's log()
// takes some sixty of its slots (C = 64, F = 8,192: 52 us for the 524,288
// logarithms of a re-fit); this one takes fourteen.  Table-driven reduction (P.
// T. P. Tang, "Table-driven implementation of the logarithm function in IEEE
// floating-point arithmetic", ACM TOMS 16, 1990): x = 2^e m, c_i = 1 / (1 + (i +
// 1/2) / 128) rounded to 16 bits for the leading seven bits i of m, r = m c_i -
// 1 with |r| <= 2^-8, and log x = e ln 2 - log c_i + log(1 + r).  The series of
// log(1 + r) is taken to r^6 (the next term is below 2^-58), its terms from r^4
// on in FP32 (|r^4 / 4| <= 2^-34, so their rounding is below 2^-57); ln 2 is
// split so that e times its high part is exact.  Over 100,000 arguments against
// 60 decimals: within 0.68 units in the last place for |log x| >= 1 and 0.62
// for |log x| >= 4; 1.1e-16 absolute below 1 (log 1 = 0 exactly).
#pragma once

#include <cuda_runtime.h>

namespace nbg {

struct Log64Entry {
  double c, l;   // c_i and -log c_i
};

static __device__ const Log64Entry kLog64[128] = {
    {0x1.fe02000000000p-1, 0x1.fefeaa2b11bc0p-9}, {0x1.fa12000000000p-1, 0x1.7db6f5f8c6e76p-7},
    {0x1.f632000000000p-1, 0x1.3ccb043c0b74dp-6}, {0x1.f260000000000p-1, 0x1.b9e8027e1918ep-6},
    {0x1.ee9c000000000p-1, 0x1.1b15d8934dd83p-5}, {0x1.eae8000000000p-1, 0x1.58a63afc8f4d5p-5},
    {0x1.e742000000000p-1, 0x1.95c290ed0ccebp-5}, {0x1.e3aa000000000p-1, 0x1.d26758b16243fp-5},
    {0x1.e01e000000000p-1, 0x1.075993598e4f1p-4}, {0x1.dca0000000000p-1, 0x1.254062f0a9417p-4},
    {0x1.d930000000000p-1, 0x1.42e64bec266e7p-4}, {0x1.d5ca000000000p-1, 0x1.606c5a94e854ap-4},
    {0x1.d272000000000p-1, 0x1.7dae56d932353p-4}, {0x1.cf26000000000p-1, 0x1.9abc1463fb437p-4},
    {0x1.cbe6000000000p-1, 0x1.b79412bcd862ap-4}, {0x1.c8b2000000000p-1, 0x1.d434cd6730bdep-4},
    {0x1.c58a000000000p-1, 0x1.f09cbc0254f21p-4}, {0x1.c26c000000000p-1, 0x1.066e412d3ba6cp-3},
    {0x1.bf58000000000p-1, 0x1.14797846886adp-3}, {0x1.bc50000000000p-1, 0x1.22663190aeacbp-3},
    {0x1.b952000000000p-1, 0x1.303ce98e4c813p-3}, {0x1.b65e000000000p-1, 0x1.3dfd030ed7c6ap-3},
    {0x1.b374000000000p-1, 0x1.4ba5df3a046e7p-3}, {0x1.b094000000000p-1, 0x1.5936dd9a31989p-3},
    {0x1.adbe000000000p-1, 0x1.66af5c2791592p-3}, {0x1.aaf2000000000p-1, 0x1.740eb7540ede5p-3},
    {0x1.a82e000000000p-1, 0x1.815df2146fa2bp-3}, {0x1.a574000000000p-1, 0x1.8e92dde888641p-3},
    {0x1.a2c2000000000p-1, 0x1.9bb69ae8857c6p-3}, {0x1.a01a000000000p-1, 0x1.a8bed7c882f59p-3},
    {0x1.9d7a000000000p-1, 0x1.b5b4d1e8fc9e4p-3}, {0x1.9ae2000000000p-1, 0x1.c2980d58e7101p-3},
    {0x1.9852000000000p-1, 0x1.cf680ce200a25p-3}, {0x1.95cc000000000p-1, 0x1.dc1a3a0ae5d7dp-3},
    {0x1.934c000000000p-1, 0x1.e8c2352ae9b61p-3}, {0x1.90d4000000000p-1, 0x1.f55575662a440p-3},
    {0x1.8e66000000000p-1, 0x1.00e4985b6bf39p-2}, {0x1.8bfc000000000p-1, 0x1.071dddfd85591p-2},
    {0x1.899c000000000p-1, 0x1.0d46dd79ac3cbp-2}, {0x1.8742000000000p-1, 0x1.1369b4296dcd1p-2},
    {0x1.84f0000000000p-1, 0x1.1980f2dd42b6fp-2}, {0x1.82a4000000000p-1, 0x1.1f91a1e4e1f74p-2},
    {0x1.8060000000000p-1, 0x1.2596410df963ap-2}, {0x1.7e22000000000p-1, 0x1.2b93e7aba3345p-2},
    {0x1.7bec000000000p-1, 0x1.31850495d0602p-2}, {0x1.79ba000000000p-1, 0x1.37742a2c6147dp-2},
    {0x1.7790000000000p-1, 0x1.3d565a5c5bf10p-2}, {0x1.756c000000000p-1, 0x1.4330caa0bb496p-2},
    {0x1.7350000000000p-1, 0x1.48fdc804dd1cbp-2}, {0x1.7138000000000p-1, 0x1.4ec8232637469p-2},
    {0x1.6f26000000000p-1, 0x1.548a303add283p-2}, {0x1.6d1a000000000p-1, 0x1.5a43bf0f72302p-2},
    {0x1.6b14000000000p-1, 0x1.5ff49f0aca855p-2}, {0x1.6914000000000p-1, 0x1.659c9f3072a73p-2},
    {0x1.671a000000000p-1, 0x1.6b3b8e2359e5ep-2}, {0x1.6524000000000p-1, 0x1.70d6f62880abdp-2},
    {0x1.6336000000000p-1, 0x1.76633523f72edp-2}, {0x1.614c000000000p-1, 0x1.7beb98a42183cp-2},
    {0x1.5f66000000000p-1, 0x1.817005da200b6p-2}, {0x1.5d86000000000p-1, 0x1.86ea85a3716c1p-2},
    {0x1.5bac000000000p-1, 0x1.8c5ae4859690ap-2}, {0x1.59d6000000000p-1, 0x1.91c6dab45ea5ep-2},
    {0x1.5806000000000p-1, 0x1.97285811a3b76p-2}, {0x1.563a000000000p-1, 0x1.9c85242e0d181p-2},
    {0x1.5472000000000p-1, 0x1.a1dd224d82fb6p-2}, {0x1.52b0000000000p-1, 0x1.a72a2966be1eap-2},
    {0x1.50f2000000000p-1, 0x1.ac72182594a04p-2}, {0x1.4f38000000000p-1, 0x1.b1b4d0ecf3e64p-2},
    {0x1.4d84000000000p-1, 0x1.b6ec11d3dfbdep-2}, {0x1.4bd4000000000p-1, 0x1.bc1dd0b0dc58ap-2},
    {0x1.4a28000000000p-1, 0x1.c149ef115f227p-2}, {0x1.4880000000000p-1, 0x1.c6704e4016ff8p-2},
    {0x1.46dc000000000p-1, 0x1.cb90cf45cf351p-2}, {0x1.453e000000000p-1, 0x1.d0a506e750384p-2},
    {0x1.43a2000000000p-1, 0x1.d5b965ae6d1a5p-2}, {0x1.420c000000000p-1, 0x1.dac12be35a5d1p-2},
    {0x1.4078000000000p-1, 0x1.dfc8e990777b5p-2}, {0x1.3ee8000000000p-1, 0x1.e4ca2a87b390ep-2},
    {0x1.3d5e000000000p-1, 0x1.e9be5a59bbf15p-2}, {0x1.3bd6000000000p-1, 0x1.eeb238640ed14p-2},
    {0x1.3a52000000000p-1, 0x1.f39f37c82987cp-2}, {0x1.38d2000000000p-1, 0x1.f885376ff49e2p-2},
    {0x1.3756000000000p-1, 0x1.fd64160f78f92p-2}, {0x1.35dc000000000p-1, 0x1.01212712ecfcep-1},
    {0x1.3468000000000p-1, 0x1.038946fd01c3bp-1}, {0x1.32f6000000000p-1, 0x1.05f0f9d26aeacp-1},
    {0x1.3188000000000p-1, 0x1.0854e084e8e0dp-1}, {0x1.301c000000000p-1, 0x1.0ab847ed10913p-1},
    {0x1.2eb4000000000p-1, 0x1.0d17c8cc368fdp-1}, {0x1.2d50000000000p-1, 0x1.0f7351c9fcd7fp-1},
    {0x1.2bf0000000000p-1, 0x1.11cad1789b0f8p-1}, {0x1.2a92000000000p-1, 0x1.1421a4524c755p-1},
    {0x1.2938000000000p-1, 0x1.167452bb4470ap-1}, {0x1.27e0000000000p-1, 0x1.18c640ff75f06p-1},
    {0x1.268c000000000p-1, 0x1.1b13ef58506dcp-1}, {0x1.253a000000000p-1, 0x1.1d60c9e67bc93p-1},
    {0x1.23ec000000000p-1, 0x1.1fa948b8a6f8bp-1}, {0x1.22a0000000000p-1, 0x1.21f0dfc65ceecp-1},
    {0x1.2158000000000p-1, 0x1.2433fef4a4a33p-1}, {0x1.2012000000000p-1, 0x1.26762213430f0p-1},
    {0x1.1ed0000000000p-1, 0x1.28b3b0dfceb80p-1}, {0x1.1d90000000000p-1, 0x1.2af02f02be4abp-1},
    {0x1.1c52000000000p-1, 0x1.2d2b9612f502ep-1}, {0x1.1b18000000000p-1, 0x1.2f62419513e46p-1},
    {0x1.19e0000000000p-1, 0x1.3197c0fa80e6ap-1}, {0x1.18ac000000000p-1, 0x1.33c867a3f01cdp-1},
    {0x1.1778000000000p-1, 0x1.35fb76dd8c7a2p-1}, {0x1.1648000000000p-1, 0x1.382997e61da84p-1},
    {0x1.151c000000000p-1, 0x1.3a52b7e80e639p-1}, {0x1.13f0000000000p-1, 0x1.3c7e30002960cp-1},
    {0x1.12c8000000000p-1, 0x1.3ea491372685fp-1}, {0x1.11a4000000000p-1, 0x1.40c5c888eb121p-1},
    {0x1.1080000000000p-1, 0x1.42e946de080bfp-1}, {0x1.0f5e000000000p-1, 0x1.450b4b13e99a0p-1},
    {0x1.0e40000000000p-1, 0x1.472803f35eaaep-1}, {0x1.0d24000000000p-1, 0x1.49432c3a40c48p-1},
    {0x1.0c0a000000000p-1, 0x1.4b5cbc95a1d05p-1}, {0x1.0af2000000000p-1, 0x1.4d74ada47b399p-1},
    {0x1.09de000000000p-1, 0x1.4f871df513f78p-1}, {0x1.08ca000000000p-1, 0x1.519bb60c233dap-1},
    {0x1.07ba000000000p-1, 0x1.53aab65b9a60dp-1}, {0x1.06ac000000000p-1, 0x1.55b7f14ba740bp-1},
    {0x1.059e000000000p-1, 0x1.57c749343bf28p-1}, {0x1.0494000000000p-1, 0x1.59d0e6600b2c0p-1},
    {0x1.038c000000000p-1, 0x1.5bd8a70e9dab4p-1}, {0x1.0286000000000p-1, 0x1.5dde837161f34p-1},
    {0x1.0182000000000p-1, 0x1.5fe273ad2a1a9p-1}, {0x1.0080000000000p-1, 0x1.61e46fda56467p-1},
};

__device__ __forceinline__ double log64(double x) {
  const int hi = __double2hiint(x);
  if (hi < 0x00100000 || hi >= 0x7FF00000) return log(x);   // subnormal, zero, negative, inf, NaN
  const double m = __hiloint2double((hi & 0x000FFFFF) | 0x3FF00000, __double2loint(x));
  const double2 t = __ldg(reinterpret_cast<const double2*>(kLog64) + ((hi >> 13) & 127));
  const double e = (double)((hi >> 20) - 1023);
  const double r = fma(m, t.x, -1.0);
  const float f = (float)r, f2 = f * f;
  const float tail = f2 * f2 * fmaf(f, fmaf(f, -1.f / 6.f, 0.2f), -0.25f);
  const double r2 = r * r;
  double s = fma(r2, fma(r, 1.0 / 3.0, -0.5), (double)tail);   // log(1 + r) - r
  s = fma(e, 7.371002565167799e-13, s + r);   // low part of ln 2
  return fma(e, 0.6931471805592082, t.y + s);   // high part: 40 bits, the product exact
}

}  // namespace nbg
