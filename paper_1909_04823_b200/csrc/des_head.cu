// A fixed read-out that stands for the rest of the model — the layers above the first FC layer in Section
// 4.3 / Fig. 4, which the sparse path does not contain.  It turns the aggregated results of one forward into
// one logit per sample and the log loss into the upstream gradients des_backward_update consumes, so that
// multi-step runs and the closed-loop benchmark need no gradients from outside.  Nothing in it is trained.
//   logit = b0 + c_lr R_lr + c_fm fm2 + <u, relu(Z + b1)> + <q, pooled> + <d, xdense>
//   p = sigmoid(logit);  loss_b = -(y log p + (1 - y) log(1 - p));  g = (p - y) / B
//   gL = c_lr g;  gF = c_fm g;  gZ = g u [Z + b1 > 0];  gE = g q
// 8 / T warps per sample, T samples a block: the dot products are taken in double (lanes stride over the row, then a butterfly, then the
// warps in order), the gradient rows are written with 16-byte stores.
#include "des_internal.cuh"

#define HEAD_U 8
// ONE: a warp per sample (T = 8).
template <bool ONE>
__global__ void __launch_bounds__(256) head_kernel(
    int B, int k, int H, int FK, int nd, int T, uint32_t ops, float b0, float c_lr, float c_fm, const float* __restrict__ u,
    const float* __restrict__ b1, const float* __restrict__ q, const float* __restrict__ d,
    const float* __restrict__ out_small, const float* __restrict__ Z, const float* __restrict__ pooled,
    const float* __restrict__ xdense, const float* __restrict__ y, float* __restrict__ logit, float* __restrict__ loss,
    float* __restrict__ gL, float* __restrict__ gF, float* __restrict__ gZ, float* __restrict__ gE) {
  des_pdl_wait(u, b1, q, d, out_small, Z, pooled, xdense, y, logit, loss, gL, gF, gZ, gE);
  __shared__ double s_acc[8];
  const int warp = threadIdx.x >> 5, wps = ONE ? 1 : 8 / T, ws = ONE ? 0 : warp % wps;   // warps of a sample, warp within the sample
  const int lane = ws * 32 + (threadIdx.x & 31), lanes = wps * 32;     // lane and lanes of the sample
  const int b = ONE ? blockIdx.x * 8 + warp : blockIdx.x * T + warp / wps;
  const bool live = b < B;
  if (ONE && !live) return;                            // whole warp (no barrier follows)
  const int stride = k + 4;
  const bool use_z = (ops & DES_OP_DENSE1) && Z && u && b1;
  const bool use_p = (ops & DES_OP_POOL) && !(ops & DES_OP_DENSE1) && pooled && q;
  // (read before the block's barrier: an output may share memory with its input)
  const double yy = live ? (double)y[b] : 0.0;
  const double r_lr = live && (ops & DES_OP_LR) ? (double)out_small[(size_t)b * stride + k] : 0.0;
  const double r_fm = live && (ops & DES_OP_FM) ? (double)out_small[(size_t)b * stride + k + 1] : 0.0;
  double acc = 0.0;
  // Z, b1 and u of HEAD_U lanes' worth of units are fetched together (u regardless of the unit being on: a load behind the test
  // waited for it, a chain of two loads per 32 units: 777 x 400 8.1 -> 6.6 us, with four warps a sample
  // 5.5; 8192 x 256 14.2 -> 12.  The logit's double exponentials taken by one warp for the block's eight samples: 8.0 and 12.1, two
  // barriers)
  if (use_z && live) {
    const float* z = Z + (size_t)b * H;
    for (int h0 = lane; h0 < H; h0 += lanes * HEAD_U) {
      float a[HEAD_U], uu[HEAD_U];
#pragma unroll
      for (int q = 0; q < HEAD_U; ++q) {
        const int h = h0 + q * lanes;
        a[q] = 0.f; uu[q] = 0.f;
        if (h < H) { a[q] = z[h] + __ldg(b1 + h); uu[q] = __ldg(u + h); }
      }
#pragma unroll
      for (int q = 0; q < HEAD_U; ++q) if (a[q] > 0.f) acc += (double)uu[q] * (double)a[q];
    }
  }
  if (use_p && live) {
    const float4* p4 = reinterpret_cast<const float4*>(pooled + (size_t)b * FK);
    const float4* q4 = reinterpret_cast<const float4*>(q);
#pragma unroll 4
    for (int i = lane; i < FK / 4; i += lanes) {
      const float4 v = p4[i], w = __ldg(q4 + i);
      acc += (double)v.x * (double)w.x + (double)v.y * (double)w.y + (double)v.z * (double)w.z + (double)v.w * (double)w.w;
    }
  }
  if (d && xdense && live)
    for (int i = lane; i < nd; i += lanes) acc += (double)__ldg(d + i) * (double)xdense[(size_t)b * nd + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
  if (!ONE) {                                          // (all warps of the block)
    if ((threadIdx.x & 31) == 0) s_acc[warp] = acc;
    __syncthreads();
    if (!live) return;
    acc = 0.0;
    for (int i = 0; i < wps; ++i) acc += s_acc[warp - ws + i];
  }
  double zl = (double)b0 + acc;
  if (ops & DES_OP_LR) zl += (double)c_lr * r_lr;
  if (ops & DES_OP_FM) zl += (double)c_fm * r_fm;
  const double sp_neg = log1p(exp(-fabs(zl))) + (zl < 0.0 ? -zl : 0.0);   // -log p, without overflow
  const double p = 1.0 / (1.0 + exp(-zl));
  const float g = (float)((p - yy) / (double)B);
  if (lane == 0) {
    logit[b] = (float)zl;
    loss[b] = (float)(yy * sp_neg + (1.0 - yy) * (sp_neg + zl));
    if (gL) gL[b] = (ops & DES_OP_LR) ? c_lr * g : 0.f;
    if (gF) gF[b] = (ops & DES_OP_FM) ? c_fm * g : 0.f;
  }
  if (use_z && gZ) {
    const float* z = Z + (size_t)b * H;
    float* o = gZ + (size_t)b * H;
#pragma unroll 8
    for (int h = lane; h < H; h += lanes) {
      const float uu = __ldg(u + h);
      o[h] = (z[h] + __ldg(b1 + h) > 0.f) ? g * uu : 0.f;
    }
  }
  if (use_p && gE) {
    const float4* q4 = reinterpret_cast<const float4*>(q);
    float4* o = reinterpret_cast<float4*>(gE + (size_t)b * FK);
    for (int i = lane; i < FK / 4; i += lanes) {
      const float4 w = __ldg(q4 + i);
      o[i] = make_float4(g * w.x, g * w.y, g * w.z, g * w.w);
    }
  }
}

extern "C" des_status_t des_head(des_table_t* t, uint32_t ops, int32_t batch, const des_head_t* head,
                                 const des_outputs_t* out, const float* d_xdense, const float* d_y, float* d_logit,
                                 float* d_loss, const des_head_grads_t* g, void* stream) {
  if (!t || !head || !out || !d_y || !d_logit || !d_loss || !g || (ops & ~15u) || ops == 0) return DES_ERR_INVALID_ARG;
  if (batch <= 0 || batch > t->max_batch) return DES_ERR_INVALID_ARG;
  if ((ops & (DES_OP_LR | DES_OP_FM)) && !out->out_small) return DES_ERR_INVALID_ARG;
  if ((ops & DES_OP_LR) && !g->gL) return DES_ERR_INVALID_ARG;
  if ((ops & DES_OP_FM) && !g->gF) return DES_ERR_INVALID_ARG;
  if ((ops & DES_OP_DENSE1) && (!t->H || !out->Z || !head->u || !head->b1 || !g->gZ)) return DES_ERR_INVALID_ARG;
  if ((ops & DES_OP_POOL) && !(ops & DES_OP_DENSE1) && (!out->pooled || !head->q || !g->gE)) return DES_ERR_INVALID_ARG;
  if (head->n_dense < 0 || (head->n_dense > 0 && head->d && !d_xdense)) return DES_ERR_INVALID_ARG;
  cudaStream_t cs = (cudaStream_t)stream;
  des_api_begin(t, cs);
  // one warp per sample once there are samples for the chip, more below that as long as each has its rounds
  const int cols = (ops & DES_OP_DENSE1) ? (int)t->H : (ops & DES_OP_POOL) ? (int)(t->F * t->k) / 4 : 0;
  int T = 8;
  while (T > 1 && batch * (8 / T) < t->sm_count * 16 && cols >= 64 * (8 / T)) T >>= 1;
  des_launch(T == 8 ? head_kernel<true> : head_kernel<false>, (batch + T - 1) / T, 256, 0, cs, batch, (int)t->k, (int)t->H, (int)(t->F * t->k), head->n_dense, T, ops, head->b0,
             head->c_lr, head->c_fm, head->u, head->b1, head->q, head->n_dense > 0 ? head->d : nullptr, out->out_small, out->Z,
             out->pooled, d_xdense, d_y, d_logit, d_loss, g->gL, g->gF, g->gZ, g->gE);
  DES_LAUNCH_CHECK(t, "head_kernel");
  return DES_OK;
}
