// grp_riemann_batch: independent leading-term Riemann problems of the ideal
// gas solved in bulk with the solver of the flux kernel (exact solver of
// Section 2: Newton on the star pressure, relative change below rtol plus
// one more iteration), from a chosen Newton start.  It serves users who need
// the exact solver alone, and measures what each start costs in iterations.
#include <cuda_runtime.h>
#include <math.h>

#include "grp_device.cuh"
#include "grprec.h"

using namespace grp;

namespace {

// A block solves its problems grouped by wave pattern and jump: a warp takes both
// branches of a side's pressure function in every iteration when its lanes
// disagree, and waits for its slowest lane (the FP64 pipe is held as long by one
// lane as by 32).  The pattern is an FP32 estimate; it orders the work and
// changes no result.  200,003 problems: 575 us in the given order, 484 us so;
// 1,000,000: 2,668 and 2,075 us.  Small batches are cut into small blocks, one warp
// each at up to two warps per SM (9,000 problems 69 -> 64 us), so that the FP64
// units of all SMs share them: 40,000 take 138 us in blocks of 128, 165 in blocks
// of 512; from 77,824 on the order over 256 is worth more.
constexpr int RB = 256, KEYS = 16;

// 0..15: left wave, right wave (0 rarefaction, 1 shock) and the size of the jump
__device__ __forceinline__ int wave_key(const Phys& ph, const double* l, const double* r)
{
  const float g = (float)ph.gamma, gm1 = g - 1.0f;
  const float rl = (float)l[0], rr = (float)r[0], ul = (float)l[1] / rl, ur = (float)r[1] / rr;
  const float pl = gm1 * ((float)l[2] - 0.5f * (float)l[1] * ul), pr = gm1 * ((float)r[2] - 0.5f * (float)r[1] * ur);
  const float cl = sqrtf(g * pl / rl), cr = sqrtf(g * pr / rr), du = ur - ul;
  // the velocity function at p: its sign at pl and pr says on which side of them p* lies
  const bool lowl = pl < pr;
  const float pk = lowl ? pr : pl, p0 = lowl ? pl : pr, r0 = lowl ? rl : rr, c0 = lowl ? cl : cr, ck = lowl ? cr : cl;
  const float fs = (pk - p0) * sqrtf(2.0f / (r0 * ((g + 1.0f) * pk + gm1 * p0)));          // shock from p0 to pk
  const float x = __powf(p0 / pk, 0.5f * gm1 / g), fr = 2.0f * ck / gm1 * (x - 1.0f);       // rarefaction from pk to p0
  const int two = fs + du < 0.0f ? 3 : fr + du > 0.0f ? 0 : (lowl ? 1 : 2);
  const float s = fabsf(du) / (cl + cr) + fabsf(__logf(pl / pr)) * 0.2f;
  const int size = s < 0.3f ? 0 : s < 0.8f ? 1 : s < 1.5f ? 2 : 3;
  return two * 4 + size;
}

template <bool G75>
__global__ void __launch_bounds__(RB) k_riemann_batch(Phys ph, long long n, const double* __restrict__ QL,
                                                      const double* __restrict__ QR,
                                                      const double* __restrict__ p_start, double* __restrict__ ps,
                                                      int* __restrict__ iters, int* __restrict__ status,
                                                      unsigned char* __restrict__ used)
{
  __shared__ int count[KEYS], order[RB];
  const long long base = (long long)blockIdx.x * blockDim.x, j = base + threadIdx.x;
  if (threadIdx.x < KEYS) count[threadIdx.x] = 0;
  __syncthreads();
  int key = 0, rank = 0;
  if (j < n) {
    const double l[3] = {QL[j], QL[n + j], QL[2 * n + j]}, r[3] = {QR[j], QR[n + j], QR[2 * n + j]};
    key = wave_key(ph, l, r);
    rank = atomicAdd(&count[key], 1);
  }
  __syncthreads();
  if (j < n) {
    int before = 0;
    for (int k = 0; k < key; ++k) before += count[k];
    order[before + rank] = threadIdx.x;
  }
  __syncthreads();
  if (j >= n) return;
  const long long i = base + order[threadIdx.x];
  const double l[3] = {QL[i], QL[n + i], QL[2 * n + i]};
  const double r[3] = {QR[i], QR[n + i], QR[2 * n + i]};
  int st, it = 0;
  double p = 0.0;
  bool by_net = false;
  if (p_start) {
    // explicit start; PVRS when it fails
    const Side L = make_side(ph, l), R = make_side(ph, r);
    double us;
    st = star_pressure<G75>(ph, L, R, p_start[i], p, us, it);
    if (st == ST_NO_CONV) {
      int it2 = 0;
      Phys pv = ph;
      pv.guess = 0;
      st = star_pressure<G75>(pv, L, R, 0.0, p, us, it2);
      it += it2;
    }
  } else {
    RSInfo info;
    double Q[3];
    Prim W;
    st = riemann_state<G75>(ph, l, r, true, Q, W, it, &info);
    p = info.ps;
    by_net = info.guess == 1;
  }
  ps[i] = st == ST_OK ? p : 0.0;
  iters[i] = it;
  status[i] = st;
  if (used) used[i] = by_net ? 1 : 0;
}

}  // namespace

extern "C" int grp_riemann_batch(double gamma, int guess, double newton_rtol, int newton_max_iter,
                                 const float* weights, const float* box, long long n, const double* QL,
                                 const double* QR, const double* p_start, double* ps, int* iters, int* status,
                                 unsigned char* used, void* stream)
{
  if (!(gamma > 1.0 && isfinite(gamma)) || guess < GRP_GUESS_PVRS || guess > GRP_GUESS_MLP) return GRP_E_INVALID_ARG;
  if (!(newton_rtol > 0.0) || newton_max_iter < 2 || n < 0) return GRP_E_INVALID_ARG;
  if (guess == GRP_GUESS_MLP && (!weights || !box)) return GRP_E_NO_MODEL;
  if (n == 0) return GRP_OK;
  if (!QL || !QR || !ps || !iters || !status) return GRP_E_INVALID_ARG;
  Phys ph = make_phys(0.0, gamma, newton_rtol, newton_max_iter, guess);
  ph.mlp_w = guess == GRP_GUESS_MLP ? weights : nullptr;
  ph.mlp_box = guess == GRP_GUESS_MLP ? box : nullptr;
  ph.features = guess == GRP_GUESS_MLP ? 1 : 0;
  const unsigned tpb = n <= 152 * 64 ? 32u : n <= 152 * 512 ? 128u : RB;
  const unsigned nb = (unsigned)((n + tpb - 1) / tpb);
  if (gamma == 1.4)
    k_riemann_batch<true><<<nb, tpb, 0, (cudaStream_t)stream>>>(ph, n, QL, QR, p_start, ps, iters, status, used);
  else
    k_riemann_batch<false><<<nb, tpb, 0, (cudaStream_t)stream>>>(ph, n, QL, QR, p_start, ps, iters, status, used);
  return cudaGetLastError() == cudaSuccess ? GRP_OK : GRP_E_CUDA;
}
