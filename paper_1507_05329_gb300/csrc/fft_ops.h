// The compiled lengths and their launch functions (host side of fft_ct.cuh).
#pragma once
#include "cola_internal.h"

#ifndef COLA_CT_PARTS
#define COLA_CT_PARTS 16
#endif

namespace cola {

// Every launch covers a whole n^3 field (rows of pc complex entries); see fft_ct.cuh for the passes.
struct FftOps {
  int n;
  void (*r2c)(int kind, const void* const* src, int fields, long long rs, float scale, float2* const* dst,
              const FftTables&, unsigned long long* mass_acc, cudaStream_t);
  void (*c2r)(float2* const* data, int fields, const FftTables&, cudaStream_t);
  void (*c2r_dense)(const float2* data, float scale, float* out, const FftTables&, cudaStream_t);
  void (*pencils)(int axis, int dir, float2* const* data, int fields, const FftTables&, cudaStream_t);
  void (*x_mul)(const float2* src, const IcMul& mul, float2* dst, const FftTables&, cudaStream_t);   // null where ic_x is not
  void (*green)(const float2* in, float2* out_f, float2* out_h, const float* dtab, float g_scale, const FftTables&,
                float2* spec_out, cudaStream_t);
  // 2LPT fields (ic_x is null, and none of these is called, above 1024); see fft_ct.cuh
  void (*ic_x)(const float2* in, float2* const* out, int fields, float scale, const float* amp_m2, const FftTables&,
               cudaStream_t);
  void (*ic_y)(const float2* in, float2* const* out, int fields, const int* zp, const FftTables&, cudaStream_t);
  void (*ic_z1)(float2* const* t, float2* src_k, float* psi1, float r_scale, const FftTables&, cudaStream_t);
  void (*ic_z2)(float2* const* f, const float* psi1, float* psi2, float* s, float* v, float r_scale, float d1, float d2,
                const FftTables&, cudaStream_t);
  void (*lpt_adj)(const float2* const* h, const float2* const* p, float2* out, float r_scale, const float* amp_m2,
                  const FftTables&, cudaStream_t);
  void (*grad_adj)(float2* const* l, float2* out, const float* dtab, float g_scale, const FftTables&, cudaStream_t);
  void (*pencils_yz)(const float2* h, float2* out_y, float2* out_z, const float* dtab, const FftTables&, cudaStream_t);
};

namespace ct {

// Every even length 2^a 3^b 5^c from 18 to 1024, and of the longer ones the mesh sides in use: 1280, 1536 and
// 2048.  Each length costs build time, not speed, so the other long ones (1080 to 2000, of which those up to 1500
// would hold a tile of 8 columns just as well) and the shortest take the run-time plans of fft_generic.cu.
#ifdef COLA_CT_TEST_SIZES
constexpr int kCtSizes[] = {COLA_CT_TEST_SIZES};
#else
constexpr int kCtSizes[] = {18,  20,  24,  30,  32,  36,  40,  48,  50,  54,  60,  64,  72,  80,  90,  96,
                            100, 108, 120, 128, 144, 150, 160, 162, 180, 192, 200, 216, 240, 250, 256, 270,
                            288, 300, 320, 324, 360, 384, 400, 432, 450, 480, 486, 500, 512, 540, 576, 600,
                            640, 648, 720, 750, 768, 800, 810, 864, 900, 960, 972, 1000, 1024, 1280, 1536, 2048};
#endif
constexpr int kCtCount = (int)(sizeof(kCtSizes) / sizeof(kCtSizes[0]));

template <int PART>
const FftOps* ops_in_part(int n);

}  // namespace ct
}  // namespace cola
