// Arguments of the FP64 data pass (pass64.cu).
#pragma once
#include "plan.h"

namespace gbcca {

struct Pass64 {
  const void* Z[2];
  int64_t ld[2];
  int d[2];
  const double* Phi[2];
  int nviews;
  int kc;            // columns of Phi used per view
  int phistride;     // row stride of Phi
  int64_t n;
  int NC;            // columns of W: nviews kc
  double* W;         // n x NC
  double* partGram;  // [CTA][NC x NC]
  const int32_t* labels;  // FDA, else null
  const double* Cls;      // FDA: class means times Phi (l x NC)
  int l;
  double* partCls;   // FDA: [CTA][l x NC] class sums of W, or null
  const int* done;
};

// W, its Gram (gctas partials) and, with partG, Z^T W (chunks partials; FP64
// data only): two launches.
int pass64(const Pass64& a, int dtype, int gctas, int chunks, int D, double* partG, cudaStream_t st);

}  // namespace gbcca
