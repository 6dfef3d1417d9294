// DCN cross layer under DES (Section 4.4, the paragraph on DCN) and the
// transfer-volume formulas of Sections 4.1-4.3.
//
// Cross layer: w is split along its long dimension d into S contiguous slices;
// shard s forms the scalar p_s = <x[slice s], w[slice s]> per sample, (+) adds
// the scalars in shard order, and y = x0 * (+)p + b + x.  A caller that does not ask for the p_s gets
// the unsplit sum <x, w> where the rows allow it ("rows in registers"): equal up to the order of the additions.  Both passes are
// streams over [B][d] rows, bound by memory: a row is read once per array and held in registers between the dot
// product and its use ("rows in registers" below).  Rows that are not 16-byte aligned or longer than
// CX_MAX_D, and callers that want the per-shard scalars, take the kernels with one warp per sample, which read a row twice.
#include "des_internal.cuh"

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
  return v;
}

// part[s][b] (optional), P[b], y[b][:].  Slice s = columns floor(s d / S) .. floor((s+1) d / S) - 1.
__global__ void __launch_bounds__(256) cross_forward_kernel(int B, int d, int S, const float* __restrict__ x0,
                                                            const float* __restrict__ x, const float* __restrict__ w,
                                                            const float* __restrict__ bias, float* __restrict__ part,
                                                            float* __restrict__ P, float* __restrict__ y) {
  const int lane = threadIdx.x & 31;
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (b >= B) return;
  const float* xr = x + (size_t)b * d;
  float tot = 0.f;
  for (int s = 0; s < S; ++s) {
    const int lo = (int)((long long)s * d / S), hi = (int)((long long)(s + 1) * d / S);
    float ps = 0.f;
    for (int i = lo + lane; i < hi; i += 32) ps = fmaf(__ldg(xr + i), __ldg(w + i), ps);
    ps = warp_sum(ps);
    if (part && lane == 0) part[(size_t)s * B + b] = ps;
    tot += ps;                                          // (+): shard order
  }
  if (lane == 0) P[b] = tot;
  const float* x0r = x0 + (size_t)b * d;
  float* yr = y + (size_t)b * d;
  for (int i = lane; i < d; i += 32) yr[i] = fmaf(__ldg(x0r + i), tot, __ldg(bias + i) + __ldg(xr + i));
}

// t[b] = <gY_b, x0_b>;  gx = gY + t w;  gx0 = gY P.
__global__ void __launch_bounds__(256) cross_backward_rows_kernel(int B, int d, const float* __restrict__ x0,
                                                                  const float* __restrict__ w,
                                                                  const float* __restrict__ P,
                                                                  const float* __restrict__ gY, float* __restrict__ gx0,
                                                                  float* __restrict__ gx, float* __restrict__ t_out) {
  const int lane = threadIdx.x & 31;
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (b >= B) return;
  const float* gr = gY + (size_t)b * d;
  const float* x0r = x0 + (size_t)b * d;
  float t = 0.f;
  for (int i = lane; i < d; i += 32) t = fmaf(__ldg(gr + i), __ldg(x0r + i), t);
  t = warp_sum(t);
  if (lane == 0) t_out[b] = t;
  const float p = __ldg(P + b);
  for (int i = lane; i < d; i += 32) {
    const float g = __ldg(gr + i);
    gx[(size_t)b * d + i] = fmaf(t, __ldg(w + i), g);
    gx0[(size_t)b * d + i] = g * p;
  }
}

// Column sums over a chunk of the batch: pw[c][i] = sum_b t_b x[b][i], pb[c][i] = sum_b gY[b][i].
#define CROSS_CHUNKS 64
__global__ void __launch_bounds__(128) cross_backward_cols_kernel(int B, int d, const float* __restrict__ x,
                                                                  const float* __restrict__ gY,
                                                                  const float* __restrict__ t, float* __restrict__ pw,
                                                                  float* __restrict__ pb) {
  const int i = blockIdx.x * 128 + threadIdx.x;
  const int c = blockIdx.y;
  const int per = (B + CROSS_CHUNKS - 1) / CROSS_CHUNKS;
  const int b_lo = c * per, b_hi = min(B, b_lo + per);
  if (i >= d) return;
  float aw = 0.f, ab = 0.f;
  for (int b = b_lo; b < b_hi; ++b) {
    aw = fmaf(__ldg(t + b), __ldg(x + (size_t)b * d + i), aw);
    ab += __ldg(gY + (size_t)b * d + i);
  }
  pw[(size_t)c * d + i] = aw;
  pb[(size_t)c * d + i] = ab;
}

// Chunks added in chunk order (deterministic).
__global__ void __launch_bounds__(256) cross_backward_finish_kernel(int d, const float* __restrict__ pw,
                                                                    const float* __restrict__ pb, float* __restrict__ gw,
                                                                    float* __restrict__ gb) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= d) return;
  float aw = 0.f, ab = 0.f;
  for (int c = 0; c < CROSS_CHUNKS; ++c) { aw += pw[(size_t)c * d + i]; ab += pb[(size_t)c * d + i]; }
  gw[i] = aw; gb[i] = ab;
}

// ---- rows in registers ---------------------------------------------------------------------------------
// A row is spread over TPR threads (a multiple of 32), one 16-byte column each, RG rows side by side in a block; a block
// takes CX_R rows of every group at a time, all their loads in flight together, and reduces their dot products with one
// barrier.  16384 x 1248: forward 80 -> 45 us, backward 157 -> 75 us.
#define CX_R 4
#define CX_MAX_D 2048
#define CX_BLOCKS 296          // blocks of the backward = partial column sums (two per SM of a B200)

struct CrossGeom { int d4, tpr, rg; };
static CrossGeom cross_geom(int d) {
  CrossGeom g;
  g.d4 = d / 4; g.tpr = (g.d4 + 31) / 32 * 32; g.rg = g.tpr >= 256 ? 1 : 256 / g.tpr;
  return g;
}
static bool cross_vec(int d, const void* a, const void* b, const void* c, const void* e, const void* f, const void* h) {
  return d % 4 == 0 && d <= CX_MAX_D &&
         ((((uintptr_t)a) | ((uintptr_t)b) | ((uintptr_t)c) | ((uintptr_t)e) | ((uintptr_t)f) | ((uintptr_t)h)) & 15) == 0;
}
__device__ __forceinline__ float cx_dot(const float4& a, const float4& b) {
  return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
}
// sums of v[] over a row's threads, in every one of them (s_part[2]: rounds alternate, so one barrier each suffices)
__device__ __forceinline__ void cx_sum(float (&v)[CX_R], float (*s_part)[16], int warp0, int nwarp, int wrow) {
#pragma unroll
  for (int r = 0; r < CX_R; ++r) v[r] = warp_sum(v[r]);
  if (nwarp == 1) return;                              // (the whole block: TPR = 32)
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int r = 0; r < CX_R; ++r) s_part[r][warp0 + wrow] = v[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < CX_R; ++r) {
    float a = 0.f;
    for (int i = 0; i < nwarp; ++i) a += s_part[r][warp0 + i];
    v[r] = a;
  }
}

__global__ void __launch_bounds__(512) cross_forward_rows_kernel(int B, CrossGeom cg, const float4* __restrict__ x0,
                                                                 const float4* __restrict__ x, const float4* __restrict__ w,
                                                                 const float4* __restrict__ bias, float* __restrict__ P,
                                                                 float4* __restrict__ y) {
  __shared__ float s_part[2][CX_R][16];
  des_pdl_wait(x0, x, w, bias, P, y);
  const int grp = threadIdx.x / cg.tpr, c = threadIdx.x % cg.tpr, nw = cg.tpr / 32;
  const bool act = c < cg.d4;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 w4 = act ? __ldg(w + c) : zero, b4 = act ? __ldg(bias + c) : zero;
  const int step = (int)gridDim.x * cg.rg * CX_R;
  int it = 0;
  for (int base = (int)blockIdx.x * cg.rg * CX_R; base < B; base += step, ++it) {
    const int b0 = base + grp * CX_R;
    float4 xv[CX_R], xz[CX_R];
    float v[CX_R];
#pragma unroll
    for (int r = 0; r < CX_R; ++r) {
      const bool in = act && b0 + r < B;
      const size_t o = (size_t)(b0 + r) * cg.d4 + c;
      xv[r] = in ? __ldg(x + o) : zero;
      xz[r] = in ? __ldg(x0 + o) : zero;
    }
#pragma unroll
    for (int r = 0; r < CX_R; ++r) v[r] = cx_dot(xv[r], w4);
    cx_sum(v, s_part[it & 1], grp * nw, nw, c / 32);
#pragma unroll
    for (int r = 0; r < CX_R; ++r) {
      if (b0 + r >= B) continue;
      if (c == 0) P[b0 + r] = v[r];
      if (act)
        __stcs(y + (size_t)(b0 + r) * cg.d4 + c,
               make_float4(fmaf(xz[r].x, v[r], b4.x + xv[r].x), fmaf(xz[r].y, v[r], b4.y + xv[r].y),
                           fmaf(xz[r].z, v[r], b4.z + xv[r].z), fmaf(xz[r].w, v[r], b4.w + xv[r].w)));
    }
  }
}

// t_b = <gY_b, x0_b>;  gx = gY + t w;  gx0 = gY P; and the block's sums of t_b x_b and gY_b, in row order per group, the
// groups in order: pw[block][:], pb[block][:].
__global__ void __launch_bounds__(512) cross_backward_vec_kernel(int B, CrossGeom cg, const float4* __restrict__ x0,
                                                                 const float4* __restrict__ x, const float4* __restrict__ w,
                                                                 const float* __restrict__ P, const float4* __restrict__ gY,
                                                                 float4* __restrict__ gx0, float4* __restrict__ gx,
                                                                 float4* __restrict__ pw, float4* __restrict__ pb) {
  __shared__ float s_part[2][CX_R][16];
  __shared__ float4 s_sum[2][512];
  des_pdl_wait(x0, x, w, P, gY, gx0, gx, pw, pb);
  const int grp = threadIdx.x / cg.tpr, c = threadIdx.x % cg.tpr, nw = cg.tpr / 32;
  const bool act = c < cg.d4;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 w4 = act ? __ldg(w + c) : zero;
  float4 aw = zero, ab = zero;
  const int step = (int)gridDim.x * cg.rg * CX_R;
  int it = 0;
  for (int base = (int)blockIdx.x * cg.rg * CX_R; base < B; base += step, ++it) {
    const int b0 = base + grp * CX_R;
    float4 g[CX_R], xz[CX_R], xv[CX_R];
    float v[CX_R], p[CX_R];
#pragma unroll
    for (int r = 0; r < CX_R; ++r) {
      const bool in = act && b0 + r < B;
      const size_t o = (size_t)(b0 + r) * cg.d4 + c;
      g[r] = in ? __ldg(gY + o) : zero;
      xz[r] = in ? __ldg(x0 + o) : zero;
      xv[r] = in ? __ldg(x + o) : zero;
      p[r] = b0 + r < B ? __ldg(P + b0 + r) : 0.f;
    }
#pragma unroll
    for (int r = 0; r < CX_R; ++r) v[r] = cx_dot(g[r], xz[r]);
    cx_sum(v, s_part[it & 1], grp * nw, nw, c / 32);
#pragma unroll
    for (int r = 0; r < CX_R; ++r) {
      aw.x = fmaf(v[r], xv[r].x, aw.x); aw.y = fmaf(v[r], xv[r].y, aw.y);
      aw.z = fmaf(v[r], xv[r].z, aw.z); aw.w = fmaf(v[r], xv[r].w, aw.w);
      ab.x += g[r].x; ab.y += g[r].y; ab.z += g[r].z; ab.w += g[r].w;
      if (!act || b0 + r >= B) continue;
      const size_t o = (size_t)(b0 + r) * cg.d4 + c;
      __stcs(gx + o, make_float4(fmaf(v[r], w4.x, g[r].x), fmaf(v[r], w4.y, g[r].y), fmaf(v[r], w4.z, g[r].z), fmaf(v[r], w4.w, g[r].w)));
      __stcs(gx0 + o, make_float4(g[r].x * p[r], g[r].y * p[r], g[r].z * p[r], g[r].w * p[r]));
    }
  }
  s_sum[0][threadIdx.x] = aw; s_sum[1][threadIdx.x] = ab;
  __syncthreads();
  if (grp == 0 && act) {
    for (int i = 1; i < cg.rg; ++i) {
      const float4 a = s_sum[0][i * cg.tpr + c], b = s_sum[1][i * cg.tpr + c];
      aw.x += a.x; aw.y += a.y; aw.z += a.z; aw.w += a.w; ab.x += b.x; ab.y += b.y; ab.z += b.z; ab.w += b.w;
    }
    pw[(size_t)blockIdx.x * cg.d4 + c] = aw;
    pb[(size_t)blockIdx.x * cg.d4 + c] = ab;
  }
}

// The blocks' sums added up: 8 columns a block, 32 lanes over the blocks (each in block order, then a fixed tree).
__global__ void __launch_bounds__(256) cross_backward_sums_kernel(int d, int blocks, const float* __restrict__ pw,
                                                                  const float* __restrict__ pb, float* __restrict__ gw,
                                                                  float* __restrict__ gb) {
  des_pdl_wait(pw, pb, gw, gb);
  const int c = threadIdx.x & 7, part = threadIdx.x >> 3, i = blockIdx.x * 8 + c;
  __shared__ float s_w[32][8], s_b[32][8];
  float aw = 0.f, ab = 0.f;
  if (i < d)
    for (int b = part; b < blocks; b += 32) { aw += __ldg(pw + (size_t)b * d + i); ab += __ldg(pb + (size_t)b * d + i); }
  s_w[part][c] = aw; s_b[part][c] = ab;
  __syncthreads();
  for (int h = 16; h > 0; h >>= 1) {
    if (part < h) { s_w[part][c] += s_w[part + h][c]; s_b[part][c] += s_b[part + h][c]; }
    __syncthreads();
  }
  if (part == 0 && i < d) { gw[i] = s_w[0][c]; gb[i] = s_b[0][c]; }
}

extern "C" int64_t des_cross_workspace_floats(int32_t batch, int32_t dim) {
  if (batch <= 0 || dim <= 0) return 0;
  return ((int64_t)batch + 3) / 4 * 4 + 2ll * (CX_BLOCKS > CROSS_CHUNKS ? CX_BLOCKS : CROSS_CHUNKS) * dim;
}

extern "C" des_status_t des_cross_forward(int32_t batch, int32_t dim, int32_t num_shards, const float* d_x0,
                                          const float* d_x, const float* d_w, const float* d_b, float* d_part,
                                          float* d_P, float* d_y, void* stream) {
  if (batch <= 0 || dim <= 0 || num_shards <= 0 || num_shards > dim || !d_x0 || !d_x || !d_w || !d_b || !d_P || !d_y)
    return DES_ERR_INVALID_ARG;
  if (!d_part && cross_vec(dim, d_x0, d_x, d_w, d_b, d_y, d_y)) {
    const CrossGeom g = cross_geom(dim);
    const int need = (batch + g.rg * CX_R - 1) / (g.rg * CX_R), most = 4 * CX_BLOCKS;
    des_launch(cross_forward_rows_kernel, need < most ? need : most, g.tpr * g.rg, 0, (cudaStream_t)stream, batch, g,
               (const float4*)d_x0, (const float4*)d_x, (const float4*)d_w, (const float4*)d_b, d_P, (float4*)d_y);
    return cudaGetLastError() == cudaSuccess ? DES_OK : DES_ERR_CUDA;
  }
  cross_forward_kernel<<<(batch + 7) / 8, 256, 0, (cudaStream_t)stream>>>(batch, dim, num_shards, d_x0, d_x, d_w, d_b,
                                                                         d_part, d_P, d_y);
  return cudaGetLastError() == cudaSuccess ? DES_OK : DES_ERR_CUDA;
}

extern "C" des_status_t des_cross_backward(int32_t batch, int32_t dim, const float* d_x0, const float* d_x,
                                           const float* d_w, const float* d_P, const float* d_gY, float* d_gx0,
                                           float* d_gx, float* d_gw, float* d_gb, float* d_ws, void* stream) {
  if (batch <= 0 || dim <= 0 || !d_x0 || !d_x || !d_w || !d_P || !d_gY || !d_gx0 || !d_gx || !d_gw || !d_gb || !d_ws)
    return DES_ERR_INVALID_ARG;
  cudaStream_t cs = (cudaStream_t)stream;
  float* t = d_ws;
  float* pw = d_ws + (batch + 3) / 4 * 4;
  if (cross_vec(dim, d_x0, d_x, d_w, d_gY, d_gx0, d_gx) && ((uintptr_t)d_ws & 15) == 0) {
    const CrossGeom g = cross_geom(dim);
    const int need = (batch + g.rg * CX_R - 1) / (g.rg * CX_R), blocks = need < CX_BLOCKS ? need : CX_BLOCKS;
    float* pb = pw + (size_t)blocks * dim;
    des_launch(cross_backward_vec_kernel, blocks, g.tpr * g.rg, 0, cs, batch, g, (const float4*)d_x0, (const float4*)d_x,
               (const float4*)d_w, d_P, (const float4*)d_gY, (float4*)d_gx0, (float4*)d_gx, (float4*)pw, (float4*)pb);
    des_launch(cross_backward_sums_kernel, (dim + 7) / 8, 256, 0, cs, dim, blocks, (const float*)pw, (const float*)pb, d_gw, d_gb);
    return cudaGetLastError() == cudaSuccess ? DES_OK : DES_ERR_CUDA;
  }
  float* pb = pw + (size_t)CROSS_CHUNKS * dim;
  cross_backward_rows_kernel<<<(batch + 7) / 8, 256, 0, cs>>>(batch, dim, d_x0, d_w, d_P, d_gY, d_gx0, d_gx, t);
  cross_backward_cols_kernel<<<dim3((dim + 127) / 128, CROSS_CHUNKS), 128, 0, cs>>>(batch, dim, d_x, d_gY, t, pw, pb);
  cross_backward_finish_kernel<<<(dim + 255) / 256, 256, 0, cs>>>(dim, pw, pb, d_gw, d_gb);
  return cudaGetLastError() == cudaSuccess ? DES_OK : DES_ERR_CUDA;
}

// Bytes a worker moves per iteration under the mesh strategy and under DES, and the saving
// ratio 1 - Q_DES / Q_Mesh, for LR, FM order 2 and the DNN first layer (Sections 4.1-4.3).
extern "C" des_status_t des_comm_volume(const des_comm_model_t* m, des_comm_volume_t* out) {
  if (!m || !out || m->workers < 2 || m->batch <= 0 || m->uniq <= 0 || m->emb_dim <= 0 || m->hidden < 0 ||
      m->key_bytes <= 0 || m->value_bytes <= 0 || m->first_layer_bytes < 0)
    return DES_ERR_INVALID_ARG;
  const double frac = (double)(m->workers - 1) / (double)m->workers;     // share held by the other workers
  const double keys = (double)m->key_bytes * (double)m->uniq;            // S_f
  const double vb = (double)m->value_bytes;
  const double weights[3] = {vb * (double)m->uniq,                                       // S_w
                             vb * (double)m->emb_dim * (double)m->uniq,                  // S_V
                             vb * (double)m->emb_dim * (double)m->uniq + m->first_layer_bytes};  // S_V + S_W
  const double partials[3] = {vb * (double)m->batch,                                     // M_1: a scalar per sample
                              vb * (double)m->batch * ((double)m->emb_dim + 1.0),        // M_1 (k-vector) + M_2
                              vb * (double)m->batch * (double)m->hidden};                // M_1 = V_i^T W_i
  for (int i = 0; i < 3; ++i) {
    out->q_mesh[i] = frac * (keys + weights[i]);
    out->q_des[i] = 2.0 * frac * partials[i];
    out->saving[i] = 1.0 - out->q_des[i] / out->q_mesh[i];
  }
  return DES_OK;
}
