// ga.cu -- one generation of the genetic algorithm that fits the minimal Tersoff parameters
// (arXiv:1909.11474, Sec. III.B): rank the population by fitness, keep the elite, keep the N_par best
// as parents, refill the population with children made by uniform crossover, mutate genes (N_pop <= 4096
// individuals of G genes each: 6 for the minimal potential, 9 for the Tersoff form); the random numbers
// are drawn by the caller and passed in.
#include <cuda_runtime.h>
#include <math.h>

#include "common.cuh"
#include "ctx.hpp"

namespace tsf {

constexpr int kGaThreads = 256;
constexpr int kGaMaxPop = 4096;
constexpr int kGaMaxGenes = 16;

// Sort key of a fitness: an unsigned integer that orders as the doubles do, with -0 = +0 and every
// non-finite Z as +infinity. (The device's FP64 unit compares a warp in 16 cycles, the integer one in 1.)
__device__ __forceinline__ unsigned long long ga_key(double z) {
  unsigned long long b = (unsigned long long)__double_as_longlong(z);
  if (((b >> 52) & 0x7ffu) == 0x7ffu) b = 0x7ff0000000000000ull;
  if ((b << 1) == 0ull) b = 0ull;
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Every CTA ranks the whole population (bitonic sort of (key, index) pairs in shared memory, padded to
// a power of two with keys behind every real one; pairs less than 32 apart stay within a warp, whose
// stages need no CTA barrier) and forms kGaThreads genes of the new population, one per thread. What
// bounds it is latency: the sort's dependent steps, then a chain of three loads and ~6 FP64 operations.
// One CTA that compared all pairs in FP64 took 31.8 us at P = 200, G = 6 and grew with P^2; back-to-back
// calls went from 32.8 to 13.8 us, where the host's launch is what is left.
__global__ void __launch_bounds__(kGaThreads) ga_step_kernel(
    int P, int G, int n_par, int np2, double rate, const double *__restrict__ Z, const double *__restrict__ genes_in,
    const double *__restrict__ u, const double *__restrict__ lo, const double *__restrict__ hi,
    double *__restrict__ genes_out, double *__restrict__ params_out, int *__restrict__ order_out) {
  __shared__ unsigned long long s_key[kGaMaxPop];
  __shared__ unsigned short s_order[kGaMaxPop];   // at most kGaMaxPop individuals
  const int tid = threadIdx.x;
  for (int i = tid; i < np2; i += kGaThreads) {
    s_key[i] = i < P ? ga_key(Z[i]) : ~0ull;
    s_order[i] = (unsigned short)i;
  }
  __syncthreads();
  for (int k = 2; k <= np2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = tid; t < (np2 >> 1); t += kGaThreads) {
        const int a = 2 * t - (t & (j - 1)), b = a + j;   // a has bit j clear
        const unsigned long long ka = s_key[a], kb = s_key[b];
        const unsigned short ia = s_order[a], ib = s_order[b];
        const bool after = ka > kb || (ka == kb && ia > ib);   // a comes after b: a strict order
        if (after == ((a & k) == 0)) {
          s_key[a] = kb;
          s_key[b] = ka;
          s_order[a] = ib;
          s_order[b] = ia;
        }
      }
      // the next stage's pairs lie in blocks of 2 j' elements, j' = its stride: a warp's 32 pairs of
      // this stage and of the next cover the same elements while both strides are at most 32
      const int jn = j > 1 ? j >> 1 : k;
      if (j <= 32 && jn <= 32) __syncwarp();
      else __syncthreads();
    }
  __syncthreads();
  const int base = (G + 2) * (P - n_par);
  const int t = blockIdx.x * kGaThreads + tid;
  if (t < P * G) {
    const int i = t / G, g = t % G;
    double v;
    if (i < n_par) {
      v = genes_in[s_order[i] * G + g];                  // elite first, then the other parents
    } else {                                             // uniform crossover of two drawn parents
      const int c = i - n_par;
      const int pa = min((int)(u[(G + 2) * c] * (double)n_par), n_par - 1);
      const int pb = min((int)(u[(G + 2) * c + 1] * (double)n_par), n_par - 1);
      const int src = u[(G + 2) * c + 2 + g] < 0.5 ? pa : pb;
      v = genes_in[s_order[src] * G + g];
    }
    if (i >= 1) {                                        // mutation, the elite excepted
      const int k = base + 2 * G * (i - 1) + 2 * g;
      if (u[k] < rate) v = u[k + 1];
    }
    genes_out[t] = v;
    params_out[t] = __dadd_rn(lo[g], __dmul_rn(v, __dsub_rn(hi[g], lo[g])));   // lo + gene (hi - lo), unfused
  }
  if (order_out && t < P) order_out[t] = s_order[t];
}

}  // namespace tsf

extern "C" int tersoff_ga_step(int32_t P, int32_t n_genes, int32_t n_par, double rate, const double *Z,
                               const double *genes_in, const double *uniforms, const double *lo, const double *hi,
                               double *genes_out, double *params_out, int32_t *order, tersoff_stream stream) {
  if (P < 1 || P > tsf::kGaMaxPop || n_par < 1 || n_par > P) return TERSOFF_E_ARG;
  if (n_genes < 1 || n_genes > tsf::kGaMaxGenes) return TERSOFF_E_ARG;
  if (!Z || !genes_in || !uniforms || !lo || !hi || !genes_out || !params_out) return TERSOFF_E_ARG;
  if (genes_in == genes_out || !(rate >= 0.0 && rate <= 1.0)) return TERSOFF_E_ARG;
  int np2 = 1;
  while (np2 < P) np2 <<= 1;
  const unsigned blocks = (unsigned)((P * n_genes + tsf::kGaThreads - 1) / tsf::kGaThreads);
  tsf::ga_step_kernel<<<blocks, tsf::kGaThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      P, n_genes, n_par, np2, rate, Z, genes_in, uniforms, lo, hi, genes_out, params_out, order);
  return tsf::launched(1) == cudaSuccess ? TERSOFF_OK : TERSOFF_E_CUDA;
}
