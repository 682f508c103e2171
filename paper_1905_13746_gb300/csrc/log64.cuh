// FP64 natural logarithm of a positive number, for the fits' tables.
//
// FP64 runs at about two lanes per clock and SM on this part and CUDA's log()
// takes some sixty of its slots (C = 64, F = 8,192: 52 us for the 524,288
// logarithms of a re-fit); this one takes thirteen.  Table-driven reduction (P.
// T. P. Tang, "Table-driven implementation of the logarithm function in IEEE
// floating-point arithmetic", ACM TOMS 16, 1990): x = 2^e m, c_i = 1 / (1 + (i +
// 1/2) / 128) rounded to 16 bits for the leading seven bits i of m, r = m c_i -
// 1 with |r| <= 2^-8, and log x = e ln 2 - log c_i + log(1 + r).  ln 2 and -log c_i
// are split into a multiple of 2^-42 and the rest: e times the one high part plus
// the other is exact, so that the result is one rounding of that sum and a low part
// of at most 2^-7, itself within 2^-59 (the series of log(1 + r) to r^7, the
// next term below 2^-66; its terms from r^5 on in FP32, r^5 / 5 < 2^-42).  Over
// 60,000 arguments against 60 digits within 0.5001 units in the last place for |log
// x| >= 1, within 5.6e-17 below (log 1 = 0 exactly).  With tables of one number each
// and the terms from r^4 on in FP32 it was within 0.68.
#pragma once

#include <cuda_runtime.h>

namespace nbg {

struct Log64Entry {
  double c, h, l;   // c_i; -log c_i as a multiple of 2^-42, and the rest
};

static __device__ const Log64Entry kLog64[128] = {
    {0x1.fe020p-1, 0x1.fefeaa2b00000p-9, 0x1.1bc049fdc0ac0p-45},
    {0x1.fa120p-1, 0x1.7db6f5f8c0000p-7, 0x1.b9d840748ca0ep-45},
    {0x1.f6320p-1, 0x1.3ccb043c10000p-6, -0x1.22cb350ddfd8dp-44},
    {0x1.f2600p-1, 0x1.b9e8027e20000p-6, -0x1.b9c9bb4f4fcfcp-44},
    {0x1.ee9c0p-1, 0x1.1b15d89350000p-5, -0x1.13ea842a027a8p-44},
    {0x1.eae80p-1, 0x1.58a63afc90000p-5, -0x1.656e6d58c041cp-46},
    {0x1.e7420p-1, 0x1.95c290ed10000p-5, -0x1.98ab7f2d35adap-44},
    {0x1.e3aa0p-1, 0x1.d26758b160000p-5, 0x1.21f91f44bb9f9p-44},
    {0x1.e01e0p-1, 0x1.0759935990000p-4, -0x1.b0ecfe4604432p-44},
    {0x1.dca00p-1, 0x1.254062f0a8000p-4, 0x1.416fe50bf3c56p-44},
    {0x1.d9300p-1, 0x1.42e64bec28000p-4, -0x1.9188e4249d675p-44},
    {0x1.d5ca0p-1, 0x1.606c5a94e8000p-4, 0x1.5292075665322p-46},
    {0x1.d2720p-1, 0x1.7dae56d934000p-4, -0x1.cac86f43c1d8cp-44},
    {0x1.cf260p-1, 0x1.9abc1463fc000p-4, -0x1.79171ca0d03a2p-45},
    {0x1.cbe60p-1, 0x1.b79412bcd8000p-4, 0x1.8a82bfd3615f0p-46},
    {0x1.c8b20p-1, 0x1.d434cd6730000p-4, 0x1.7bc9ecd3d322bp-45},
    {0x1.c58a0p-1, 0x1.f09cbc0254000p-4, 0x1.e4247e9577786p-45},
    {0x1.c26c0p-1, 0x1.066e412d3c000p-3, -0x1.650ea9f71aa62p-45},
    {0x1.bf580p-1, 0x1.1479784688000p-3, 0x1.ab21c0820b429p-45},
    {0x1.bc500p-1, 0x1.22663190ae000p-3, 0x1.596e8a3e0d005p-44},
    {0x1.b9520p-1, 0x1.303ce98e4c000p-3, 0x1.025f6c31cabb9p-44},
    {0x1.b65e0p-1, 0x1.3dfd030ed8000p-3, -0x1.cb144b686618fp-46},
    {0x1.b3740p-1, 0x1.4ba5df3a04000p-3, 0x1.b9a3c69363383p-45},
    {0x1.b0940p-1, 0x1.5936dd9a32000p-3, -0x1.9dc954aa776e5p-45},
    {0x1.adbe0p-1, 0x1.66af5c2792000p-3, -0x1.4db8e44950281p-44},
    {0x1.aaf20p-1, 0x1.740eb7540e000p-3, 0x1.bc979c6007c5bp-44},
    {0x1.a82e0p-1, 0x1.815df21470000p-3, -0x1.75256d92bec69p-45},
    {0x1.a5740p-1, 0x1.8e92dde888000p-3, 0x1.902abfd25a3dcp-45},
    {0x1.a2c20p-1, 0x1.9bb69ae886000p-3, -0x1.073c57ce45926p-44},
    {0x1.a01a0p-1, 0x1.a8bed7c882000p-3, 0x1.eb185cf770f25p-44},
    {0x1.9d7a0p-1, 0x1.b5b4d1e8fc000p-3, 0x1.3c8dc20fee737p-44},
    {0x1.9ae20p-1, 0x1.c2980d58e8000p-3, -0x1.dfe20bf067217p-44},
    {0x1.98520p-1, 0x1.cf680ce200000p-3, 0x1.44a14d7187873p-44},
    {0x1.95cc0p-1, 0x1.dc1a3a0ae6000p-3, -0x1.4178471a81993p-46},
    {0x1.934c0p-1, 0x1.e8c2352aea000p-3, -0x1.27d6ed05822d9p-45},
    {0x1.90d40p-1, 0x1.f55575662a000p-3, 0x1.101438adbd445p-45},
    {0x1.8e660p-1, 0x1.00e4985b6c000p-2, -0x1.8d4755bce7d5dp-47},
    {0x1.8bfc0p-1, 0x1.071dddfd85000p-2, 0x1.6459eebab1a3dp-44},
    {0x1.899c0p-1, 0x1.0d46dd79ac000p-2, 0x1.e5906872c81ffp-45},
    {0x1.87420p-1, 0x1.1369b4296e000p-2, -0x1.977a13c647652p-45},
    {0x1.84f00p-1, 0x1.1980f2dd43000p-2, -0x1.24262183a4308p-44},
    {0x1.82a40p-1, 0x1.1f91a1e4e2000p-2, -0x1.17dd97615905fp-47},
    {0x1.80600p-1, 0x1.2596410df9000p-2, 0x1.8e7c177a43938p-44},
    {0x1.7e220p-1, 0x1.2b93e7aba3000p-2, 0x1.a26cf6f90d899p-45},
    {0x1.7bec0p-1, 0x1.31850495d0000p-2, 0x1.807adf756f48dp-44},
    {0x1.79ba0p-1, 0x1.37742a2c61000p-2, 0x1.1f3201bc4f554p-44},
    {0x1.77900p-1, 0x1.3d565a5c5c000p-2, -0x1.df35e81128443p-47},
    {0x1.756c0p-1, 0x1.4330caa0bb000p-2, 0x1.25731cd21d67dp-44},
    {0x1.73500p-1, 0x1.48fdc804dd000p-2, 0x1.cac483712b8e4p-46},
    {0x1.71380p-1, 0x1.4ec8232637000p-2, 0x1.1a3b998405490p-44},
    {0x1.6f260p-1, 0x1.548a303add000p-2, 0x1.4167e63b2c7a2p-45},
    {0x1.6d1a0p-1, 0x1.5a43bf0f72000p-2, 0x1.8103a053d320bp-45},
    {0x1.6b140p-1, 0x1.5ff49f0acb000p-2, -0x1.eab7866daed1cp-44},
    {0x1.69140p-1, 0x1.659c9f3073000p-2, -0x1.6332aa5d24e3cp-44},
    {0x1.671a0p-1, 0x1.6b3b8e235a000p-2, -0x1.a276de1b31cc1p-46},
    {0x1.65240p-1, 0x1.70d6f62881000p-2, -0x1.50bf9e9f5b591p-44},
    {0x1.63360p-1, 0x1.76633523f7000p-2, 0x1.76992f6bc68d7p-45},
    {0x1.614c0p-1, 0x1.7beb98a422000p-2, -0x1.f115bbfb0fb3fp-44},
    {0x1.5f660p-1, 0x1.817005da20000p-2, 0x1.6bb80650a7290p-47},
    {0x1.5d860p-1, 0x1.86ea85a371000p-2, 0x1.b03fd2abdcd33p-44},
    {0x1.5bac0p-1, 0x1.8c5ae48597000p-2, -0x1.bd6281df29608p-44},
    {0x1.59d60p-1, 0x1.91c6dab45f000p-2, -0x1.689d109026758p-44},
    {0x1.58060p-1, 0x1.97285811a4000p-2, -0x1.226ec74108d28p-44},
    {0x1.563a0p-1, 0x1.9c85242e0d000p-2, 0x1.815fc660c1797p-46},
    {0x1.54720p-1, 0x1.a1dd224d83000p-2, -0x1.289de56dcc6d8p-48},
    {0x1.52b00p-1, 0x1.a72a2966be000p-2, 0x1.ea167cc070d2ep-46},
    {0x1.50f20p-1, 0x1.ac72182595000p-2, -0x1.7ef97ffd4bd53p-44},
    {0x1.4f380p-1, 0x1.b1b4d0ecf4000p-2, -0x1.9c23eec87c60cp-46},
    {0x1.4d840p-1, 0x1.b6ec11d3e0000p-2, -0x1.0890c1e66694bp-44},
    {0x1.4bd40p-1, 0x1.bc1dd0b0dc000p-2, 0x1.6290655c5eb2fp-44},
    {0x1.4a280p-1, 0x1.c149ef115f000p-2, 0x1.135665be33dc9p-45},
    {0x1.48800p-1, 0x1.c6704e4017000p-2, -0x1.f0b4f8740cb80p-52},
    {0x1.46dc0p-1, 0x1.cb90cf45cf000p-2, 0x1.a894a701c1042p-45},
    {0x1.453e0p-1, 0x1.d0a506e750000p-2, 0x1.c1c85ea97ef77p-45},
    {0x1.43a20p-1, 0x1.d5b965ae6d000p-2, 0x1.a4c05606cac18p-46},
    {0x1.420c0p-1, 0x1.dac12be35a000p-2, 0x1.7432e470d3c40p-44},
    {0x1.40780p-1, 0x1.dfc8e99077000p-2, 0x1.ed53ea14007d7p-44},
    {0x1.3ee80p-1, 0x1.e4ca2a87b4000p-2, -0x1.bc900981afbf8p-44},
    {0x1.3d5e0p-1, 0x1.e9be5a59bc000p-2, -0x1.d6ab63fc918bap-47},
    {0x1.3bd60p-1, 0x1.eeb238640f000p-2, -0x1.75e50518d1183p-45},
    {0x1.3a520p-1, 0x1.f39f37c82a000p-2, -0x1.e0ff35bc38055p-44},
    {0x1.38d20p-1, 0x1.f885376ff5000p-2, -0x1.8770c80be9465p-44},
    {0x1.37560p-1, 0x1.fd64160f79000p-2, -0x1.b9af7a8883a88p-48},
    {0x1.35dc0p-1, 0x1.01212712ed000p-1, -0x1.8c5c685540fbfp-48},
    {0x1.34680p-1, 0x1.038946fd02000p-1, -0x1.e2922697cdf6ep-44},
    {0x1.32f60p-1, 0x1.05f0f9d26b000p-1, -0x1.54009cd7853cbp-45},
    {0x1.31880p-1, 0x1.0854e084e9000p-1, -0x1.f2a1f6f545c4dp-45},
    {0x1.301c0p-1, 0x1.0ab847ed10800p-1, 0x1.1298f508bb335p-45},
    {0x1.2eb40p-1, 0x1.0d17c8cc36800p-1, 0x1.f99fe0848f447p-46},
    {0x1.2d500p-1, 0x1.0f7351c9fd000p-1, -0x1.408bf9d0a30cap-44},
    {0x1.2bf00p-1, 0x1.11cad1789b000p-1, 0x1.efa3472134995p-46},
    {0x1.2a920p-1, 0x1.1421a4524c800p-1, -0x1.563c9cc84e329p-46},
    {0x1.29380p-1, 0x1.167452bb44800p-1, -0x1.ec6bbc73ae748p-46},
    {0x1.27e00p-1, 0x1.18c640ff76000p-1, -0x1.f48f456f6e880p-46},
    {0x1.268c0p-1, 0x1.1b13ef5850800p-1, -0x1.24697d3632b89p-45},
    {0x1.253a0p-1, 0x1.1d60c9e67c000p-1, -0x1.b67f55e418cbep-44},
    {0x1.23ec0p-1, 0x1.1fa948b8a7000p-1, -0x1.d3fd7dc6f10dep-47},
    {0x1.22a00p-1, 0x1.21f0dfc65d000p-1, -0x1.141d7a46166ddp-45},
    {0x1.21580p-1, 0x1.2433fef4a4800p-1, 0x1.19b1ab8a024cbp-44},
    {0x1.20120p-1, 0x1.2676221343000p-1, 0x1.df9a55bf74e3dp-46},
    {0x1.1ed00p-1, 0x1.28b3b0dfce800p-1, 0x1.bfd5a1fd2b26fp-44},
    {0x1.1d900p-1, 0x1.2af02f02be800p-1, -0x1.aa8f71f93d81bp-44},
    {0x1.1c520p-1, 0x1.2d2b9612f5000p-1, 0x1.6dc55a092c9fcp-48},
    {0x1.1b180p-1, 0x1.2f62419514000p-1, -0x1.b9e9559a46e34p-45},
    {0x1.19e00p-1, 0x1.3197c0fa81000p-1, -0x1.95e1f20c51be4p-45},
    {0x1.18ac0p-1, 0x1.33c867a3f0000p-1, 0x1.cd715a1ae1bb7p-45},
    {0x1.17780p-1, 0x1.35fb76dd8c800p-1, -0x1.77b8331ef542fp-47},
    {0x1.16480p-1, 0x1.382997e61d800p-1, 0x1.41c4973ac4dc0p-44},
    {0x1.151c0p-1, 0x1.3a52b7e80e800p-1, -0x1.c6fa936346f8fp-45},
    {0x1.13f00p-1, 0x1.3c7e300029800p-1, -0x1.f3cf8c0d72c81p-45},
    {0x1.12c80p-1, 0x1.3ea4913726800p-1, 0x1.7b0038197a389p-47},
    {0x1.11a40p-1, 0x1.40c5c888eb000p-1, 0x1.20906c9501b38p-45},
    {0x1.10800p-1, 0x1.42e946de08000p-1, 0x1.7e040a2c943b9p-46},
    {0x1.0f5e0p-1, 0x1.450b4b13e9800p-1, 0x1.a0493905e7c05p-45},
    {0x1.0e400p-1, 0x1.472803f35e800p-1, 0x1.56e0d6e341304p-44},
    {0x1.0d240p-1, 0x1.49432c3a41000p-1, -0x1.dc2af8f0f1148p-44},
    {0x1.0c0a0p-1, 0x1.4b5cbc95a2000p-1, -0x1.7dbd4a31cf62cp-44},
    {0x1.0af20p-1, 0x1.4d74ada47b000p-1, 0x1.cc5ef3fab80d6p-44},
    {0x1.09de0p-1, 0x1.4f871df514000p-1, -0x1.0f564cc7ab8bap-46},
    {0x1.08ca0p-1, 0x1.519bb60c23000p-1, 0x1.ed15f7878bb02p-44},
    {0x1.07ba0p-1, 0x1.53aab65b9a800p-1, -0x1.f355cdb6bbe6bp-45},
    {0x1.06ac0p-1, 0x1.55b7f14ba7800p-1, -0x1.fabbbb44272b1p-44},
    {0x1.059e0p-1, 0x1.57c749343c000p-1, -0x1.afaf727dd89adp-46},
    {0x1.04940p-1, 0x1.59d0e6600b000p-1, 0x1.6024dcb75d63bp-44},
    {0x1.038c0p-1, 0x1.5bd8a70e9d800p-1, 0x1.59eee960a5c4ep-44},
    {0x1.02860p-1, 0x1.5dde837162000p-1, -0x1.9871042999a5fp-46},
    {0x1.01820p-1, 0x1.5fe273ad2a000p-1, 0x1.a8be50fc03010p-45},
    {0x1.00800p-1, 0x1.61e46fda56800p-1, -0x1.cc9ee18ba867dp-44},
};

__device__ __forceinline__ double log64(double x) {
  const int hi = __double2hiint(x);
  if (hi < 0x00100000 || hi >= 0x7FF00000) return log(x);   // subnormal, zero, negative, inf, NaN
  const double m = __hiloint2double((hi & 0x000FFFFF) | 0x3FF00000, __double2loint(x));
  const Log64Entry* t = kLog64 + ((hi >> 13) & 127);
  const double e = (double)((hi >> 20) - 1023);
  const double r = fma(m, __ldg(&t->c), -1.0);
  const float f = (float)r, f2 = f * f;
  const float tail = f2 * f2 * f * fmaf(f, fmaf(f, 1.f / 7.f, -1.f / 6.f), 0.2f);
  const double r2 = r * r;
  const double s = fma(r2, fma(r2, -0.25, fma(r, 1.0 / 3.0, -0.5)), (double)tail);   // log(1 + r) - r
  const double lo = fma(e, 0x1.ef35793c76730p-45, __ldg(&t->l));
  return fma(e, 0x1.62e42fefa3800p-1, __ldg(&t->h)) + (r + (s + lo));   // the high parts' sum is exact
}

}  // namespace nbg
