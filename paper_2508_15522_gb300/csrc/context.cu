// Context lifetime, errors, abort flag, parameter defaults and the
// read-bandwidth probe of libgridff.
#include <stdarg.h>

#include "internal.h"

gridff_status set_err(gridff_ctx* ctx, gridff_status st, const char* fmt, ...) {
  if (ctx) {
    char buf[1024];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    ctx->err = buf;
  }
  return st;
}

extern "C" {

gridff_status gridff_create(int device, void* cuda_stream, gridff_ctx** out) {
  if (!out) return GRIDFF_EINVAL;
  *out = nullptr;
  int n_dev = 0;
  if (cudaGetDeviceCount(&n_dev) != cudaSuccess || device < 0 || device >= n_dev)
    return GRIDFF_EINVAL;
  gridff_ctx* ctx = new gridff_ctx();
  ctx->device = device;
  auto fail = [&](gridff_status st) {
    gridff_destroy(ctx);
    return st;
  };
  if (cudaSetDevice(device) != cudaSuccess) return fail(GRIDFF_ECUDA);
  if (cudaDeviceGetAttribute(&ctx->n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
    return fail(GRIDFF_ECUDA);
  if (cuda_stream) {
    ctx->stream = (cudaStream_t)cuda_stream;
  } else {
    if (cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking) != cudaSuccess)
      return fail(GRIDFF_ECUDA);
    ctx->own_stream = true;
  }
  void* h = nullptr;
  if (cudaHostAlloc(&h, 64, cudaHostAllocMapped) != cudaSuccess) return fail(GRIDFF_ENOMEM);
  ctx->ctrl_host = (volatile int*)h;
  for (int i = 0; i < 16; ++i) ctx->ctrl_host[i] = 0;
  void* d = nullptr;
  if (cudaHostGetDevicePointer(&d, h, 0) != cudaSuccess) return fail(GRIDFF_ECUDA);
  ctx->ctrl_dev = (int*)d;
  if (cudaMalloc(&ctx->result_dev, 64) != cudaSuccess) return fail(GRIDFF_ENOMEM);
  if (cudaHostAlloc(&ctx->result_host, 64, cudaHostAllocDefault) != cudaSuccess) return fail(GRIDFF_ENOMEM);
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = device;
  uint64_t kept = kScratchKept;
  if (cudaMemPoolCreate(&ctx->pool, &props) != cudaSuccess ||
      cudaMemPoolSetAttribute(ctx->pool, cudaMemPoolAttrReleaseThreshold, &kept) != cudaSuccess)
    return fail(GRIDFF_ENOMEM);
  if (cudaEventCreate(&ctx->ev0) != cudaSuccess || cudaEventCreate(&ctx->ev1) != cudaSuccess)
    return fail(GRIDFF_ECUDA);
  *out = ctx;
  return GRIDFF_OK;
}

void gridff_destroy(gridff_ctx* ctx) {
  if (!ctx) return;
  cudaSetDevice(ctx->device);
  if (ctx->stream) cudaStreamSynchronize(ctx->stream);
  if (ctx->l2_limit_set) {
    // give back the persisting-L2 set-aside taken by L2-window launches
    cudaCtxResetPersistingL2Cache();
    cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, ctx->l2_prev_limit);
    cudaGetLastError();
  }
  if (ctx->ev0) cudaEventDestroy(ctx->ev0);
  if (ctx->ev1) cudaEventDestroy(ctx->ev1);
  if (ctx->result_dev) cudaFree(ctx->result_dev);
  if (ctx->result_host) cudaFreeHost(ctx->result_host);
  if (ctx->pool) cudaMemPoolDestroy(ctx->pool);
  if (ctx->ctrl_host) cudaFreeHost((void*)ctx->ctrl_host);
  if (ctx->own_stream && ctx->stream) cudaStreamDestroy(ctx->stream);
  cudaGetLastError();   // leave no error of this teardown behind
  delete ctx;
}

const char* gridff_last_error(const gridff_ctx* ctx) { return ctx ? ctx->err.c_str() : ""; }

void* gridff_stream(const gridff_ctx* ctx) { return ctx ? (void*)ctx->stream : nullptr; }

void gridff_set_abort(gridff_ctx* ctx, int value) {
  if (ctx && ctx->ctrl_host) {
    ctx->ctrl_host[0] = value;
    __sync_synchronize();
  }
}

void gridff_grid_opts_default(gridff_grid_opts* o) {
  if (!o) return;
  *o = gridff_grid_opts{};
  o->alpha = 1.5;
  o->rcut = 17.0;
  o->ewald_tol = 1e-10;
  o->ewald_rcut = 12.0;
  o->channels = GRIDFF_CH_C | GRIDFF_CH_P | GRIDFF_CH_L;
  o->storage = GRIDFF_STORE_F32;
  o->keep_f64 = 0;
}

void gridff_fire_params_default(gridff_fire_params* p) {
  if (!p) return;
  p->dt_start = 0.5f;
  p->dt_max = 2.0f;
  p->n_min = 5;
  p->f_inc = 1.1f;
  p->f_dec = 0.5f;
  p->alpha_start = 0.1f;
  p->f_alpha = 0.99f;
  p->d_max = 0.1f;
  p->f_conv = 1e-3f;
  p->clock_budget_s = 0.0;
}

double gridff_last_kernel_ms(const gridff_ctx* ctx) { return ctx ? ctx->last_ms : 0.0; }

}  // extern "C"

// Streaming read of a device buffer: each thread reads 16-byte vectors with
// a grid-stride loop (4 independent loads in flight per iteration) and folds
// them into one word so the loads are kept.
__global__ void probe_read_kernel(const float4* __restrict__ p, size_t n, int iters,
                                  float* __restrict__ sink) {
  float acc = 0.f;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (int it = 0; it < iters; ++it) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {
      float4 a = __ldg(p + i), b = __ldg(p + i + stride), c = __ldg(p + i + 2 * stride),
             d = __ldg(p + i + 3 * stride);
      acc += (a.x + b.x) + (c.x + d.x);
    }
    for (; i < n; i += stride) acc += __ldg(p + i).x;
  }
  if (acc == 123456.789f) sink[0] = acc;   // practically never: keeps the loads live
}

// Best of a few launch shapes (blocks per SM x threads), since the peak is
// the quantity of interest.
extern "C" gridff_status gridff_probe_read_bandwidth(gridff_ctx* ctx, const void* buf, size_t bytes,
                                                     int32_t iters, double* gbs_out) {
  if (!ctx || !buf || !gbs_out || iters <= 0) return set_err(ctx, GRIDFF_EINVAL, "bad argument");
  if ((bytes % 16) != 0 || ((uintptr_t)buf % 16) != 0 || bytes == 0)
    return set_err(ctx, GRIDFF_EINVAL, "buffer must be 16-byte aligned and a multiple of 16 bytes");
  GRIDFF_CUDA(ctx, cudaSetDevice(ctx->device));
  const size_t n = bytes / 16;
  float* sink = (float*)ctx->result_dev + 12;
  const int shapes[3][2] = {{8, 256}, {4, 512}, {16, 128}};
  double best = 0.0;
  for (const auto& sh : shapes) {
    const int blocks = ctx->n_sm * sh[0];
    probe_read_kernel<<<blocks, sh[1], 0, ctx->stream>>>((const float4*)buf, n, 1, sink);  // warm
    GRIDFF_CUDA(ctx, cudaEventRecord(ctx->ev0, ctx->stream));
    probe_read_kernel<<<blocks, sh[1], 0, ctx->stream>>>((const float4*)buf, n, iters, sink);
    GRIDFF_CUDA(ctx, cudaEventRecord(ctx->ev1, ctx->stream));
    GRIDFF_CUDA(ctx, cudaEventSynchronize(ctx->ev1));
    GRIDFF_CUDA(ctx, cudaGetLastError());
    float ms = 0.f;
    GRIDFF_CUDA(ctx, cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1));
    const double gbs = (double)bytes * iters / (ms * 1e-3) / 1e9;
    if (gbs > best) best = gbs;
  }
  *gbs_out = best;
  return GRIDFF_OK;
}
