// Launch wrappers of every kernel for one (model, storage) pair.
#pragma once

#include <utility>

#include "lb_aux.cuh"
#include "lb_device.cuh"
#include "lb_ops.h"
#include "lb_step_tma.cuh"

namespace lbk {

template <class S>
static Buf<S> to_buf(const OpBufs& b, const OpArgs& a) {
  return Buf<S>{(typename S::T*)b.f, (typename S::T*)b.g, b.g0, rest_offsets_binary(a.Acoef)};
}

static inline Geom to_geom(const OpArgs& a) {
  return Geom{a.nx, a.ny, a.tube_x0, a.tube_len, a.tube_y0, a.tube_h};
}

template <typename A>
static Phys<A> to_phys(const OpArgs& a, bool lg) {
  Phys<A> p;
  p.kappa = A(a.kappa); p.a = A(a.a); p.b = A(a.b); p.T = A(a.T);
  p.Acoef = A(a.Acoef); p.M = A(a.M); p.nu_l = A(a.nu_l); p.nu_g = A(a.nu_g);
  p.nu = A(a.nu); p.lambda_scale = A(a.lambda_scale); p.h = A(a.h);
  p.lut = A(a.lut);
  p.lut_inv = a.lut > 0 ? A(1.0 / a.lut) : A(0);
  set_pair_constants(p, a.kappa, a.M, a.nu, a.lambda_scale, lg);
  return p;
}

// Blocks of a 1-D step grid: column blocks x row bands (see tile_of_block).
static inline unsigned tiles_1d(int ncb, int ny, int yc) {
  return (unsigned)ncb * (unsigned)((ny + yc - 1) / yc);
}

// Grid of a grid-stride kernel over n items: at most 16 blocks per SM of the
// current device.
static inline int grid_for(size_t n, int threads) {
  const size_t cap = 16 * (size_t)device_sm_count();
  size_t b = (n + threads - 1) / threads;
  return (int)(b > cap ? cap : (b < 1 ? 1 : b));
}

// Launch of a kernel that may start while the previous one on the stream still runs
// (pdl_wait in lb_device.cuh); captured into a graph, the dependency becomes a
// programmatic edge.
template <class... P, class... A>
static cudaError_t launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                              A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// The sliding-window variant runs as warp strips (step_strip), but for the two cases below
// and lattices beyond the strips' 32-bit offsets.  In FP64 only bands of one
// or two rows do.  The strips form the row summaries of all three rows anew for every node,
// the window does too, and the strips' 32 lanes for 30 columns stand against its barriers: us
// per step, window -> strips, liquid-gas 1024 x 64 at two rows 19.5 -> 17.5, 1000 x 200 50.2 ->
// 48.4; 4096 x 128 at three rows 107.6 -> 113.9 (128 columns), at four 109.4 -> 115.9, at six
// 117.6 -> 110.6 (64 columns); binary 4096 x 128 at three 190.0 -> 194.5, at four 193.1 -> 199.8,
// 4097 x 128 at six 231.7 -> 191.8; liquid-gas 256 x 32 at four 19.9 -> 17.1.  Above two rows the
// best tiles on 4096 x 128 are the window's (107.6 and 190.0 against 110.6 and 191.8); on small
// lattices, and on wide ones at six rows, the strips would be faster.
constexpr int kStripRowsF64 = 2;

// A strip produces 30 columns where the shared window's warp produces 32, so at some sizes
// the strips need a second wave of CTAs while the window fits in one (16 warps an SM): there
// the planes run the window (binary us per step, strips -> window: 2304 x 128 FP32 at 128 x 4
// 11.5 -> 10.0, at 64 x 4 11.6 -> 10.5, FP16 13.4 -> 11.1; 3000 x 100 and 1536 x 200 alike).
// CTAs of 256 columns are so large that one more on some SMs counts as well (1024 x 64 at
// 256 x 1: 5.1 -> 4.5; FP64 at 256 x 2: 42.2 -> 31.2).  The liquid-gas FP32 strips, which
// hold half the values, keep the second wave cheap except in those (2304 x 128: 64 x 4 7.5,
// window 8.5; 256 x 4 9.7, 8.2).
template <int MODEL, class S, int BX>
static bool window_fills_one_wave(const OpArgs& a) {
  constexpr unsigned per = 16 / (BX / 32), cols = BX / 32 * kStripCols;
  const unsigned sms = (unsigned)device_sm_count();
  const unsigned strips = tiles_1d((a.nx + cols - 1) / cols, a.ny, a.yc), window = tiles_1d((a.nx + BX - 1) / BX, a.ny, a.yc);
  if (window > per * sms) return false;
  if (MODEL == MODEL_LG && !std::is_same<typename S::A, double>::value) return BX == 256 && strips > per * sms;
  return strips > per * sms || (BX == 256 && (strips + sms - 1) / sms > (window + sms - 1) / sms);
}

template <int MODEL, class S, int BX>
static cudaError_t launch_step(const OpArgs& a, cudaStream_t s) {
  StepArgs<MODEL, S> k;
  k.G = to_geom(a);
  k.P = to_phys<typename S::A>(a, MODEL == MODEL_LG);
  k.Q = mom_phys(a.kappa, a.Acoef, a.M, a.nu_l, a.nu_g, a.lambda_scale, a.h, a.lut);
  k.src = to_buf<S>(a.src, a);
  k.dst = to_buf<S>(a.dst, a);
  k.yc = a.yc;
  if constexpr (!is_blocked<S>::value) {
    constexpr bool F64 = std::is_same<typename S::A, double>::value;
    if ((F64 ? a.yc > kStripRowsF64 : 9ull * a.nx * a.ny >= 1ull << 32) ||  // (FP32 strips: 32-bit offsets)
        window_fills_one_wave<MODEL, S, BX>(a))
      return launch_pdl(step_kernel<MODEL, S, BX>, tiles_1d((a.nx + BX - 1) / BX, a.ny, a.yc), BX, 0, s, k);
  }
  return launch_pdl(strip_kernel<MODEL, S, BX / 32>,
                    tiles_1d((a.nx + BX / 32 * kStripCols - 1) / (BX / 32 * kStripCols), a.ny, a.yc), BX, 0, s, k);
}

// When a CTA of the staged kernel lets the next step's CTAs in: as soon as its last row is
// on its way, which hides most of their start, or only when it ends.  With CTAs that are few
// and long the former puts the next step where this one ends first, several CTAs on one SM and
// none on another.  That costs FP64 bands of six rows and more and the block storages' (from
// three rows in FP32, from six in FP16) up to half a step while the CTAs are between half of
// one and about six tenths of the resident ones an SM; beyond, and in bands of fewer rows and
// the planes, whose copies set the pace, letting them in early is the faster way or makes no
// difference.  Us per step, early -> at the end:
//   FP64         1000 x 200 binary 64 x 12 130.3 -> 85.1, liquid-gas 128 x 8 93.1 -> 65.7;  4096 x 128
//                liquid-gas 64 x 32 168.7 -> 123.9;  1000 x 200 binary 128 x 8 102.3 -> 109.6 (the worst)
//   FP32 blocks  1000 x 200 64 x 6 10.3 -> 8.3;  2304 x 128 128 x 8 11.5 -> 9.3;  704 x 40 128 x 3 4.1 -> 4.4
//   FP16 blocks  4096 x 128 128 x 10 13.9 -> 11.6;  2304 x 128 128 x 6 9.8 -> 8.5;  1536 x 60 128 x 6 6.4 -> 6.8
template <class S, int BX>
static bool early_trigger(const OpArgs& a, unsigned grid) {
  constexpr bool F64 = std::is_same<typename S::A, double>::value;
  if (!F64 && !is_blocked<S>::value) return true;
  constexpr int rows = std::is_same<S, SF32B>::value ? 3 : 6;
  constexpr unsigned full = BX == 64 ? 5 : (BX == 128 ? 3 : 2);  // CTAs an SM
  const unsigned sms = (unsigned)device_sm_count();
  return a.yc < rows || 2 * grid < sms || grid >= full * sms;
}

template <int MODEL, class S, int BX, int NS>
static cudaError_t launch_staged(const OpArgs& a, cudaStream_t s) {
  using L = TmaLayout<MODEL, S, BX, NS>;
  static bool configured = false;  // dynamic shared memory opt-in, once per process
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(step_tma_kernel<MODEL, S, BX, NS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::BYTES);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  TmaArgs<MODEL, S> k;
  k.G = to_geom(a);
  k.P = to_phys<typename S::A>(a, MODEL == MODEL_LG);
  k.Q = mom_phys(a.kappa, a.Acoef, a.M, a.nu_l, a.nu_g, a.lambda_scale, a.h, a.lut);
  k.src = to_buf<S>(a.src, a);
  k.dst = to_buf<S>(a.dst, a);
  k.yc = a.yc;
  k.err = a.err;
  const unsigned grid = tiles_1d((a.nx + BX - 1) / BX, a.ny, a.yc);
  k.early = early_trigger<S, BX>(a, grid);
  return launch_pdl(step_tma_kernel<MODEL, S, BX, NS>, grid, BX + 32, L::BYTES, s, k);
}

template <int NW, class S>
static cudaError_t launch_moment(const OpArgs& a, cudaStream_t s) {
  MomArgs k;
  k.G = to_geom(a);
  k.Q = mom_phys(a.kappa, a.Acoef, a.M, a.nu_l, a.nu_g, a.lambda_scale, a.h, a.lut);
  k.src = a.src.f;
  k.dst = a.dst.f;
  k.yc = a.yc;
  const unsigned grid = tiles_1d((a.nx + NW * kMomCols - 1) / (NW * kMomCols), a.ny, a.yc);
  moment_step_kernel<NW, S><<<grid, NW * 32, 0, s>>>(k);
  return cudaGetLastError();
}

template <int MODEL, class S>
cudaError_t ops_impl(OpKind op, const OpArgs& a, cudaStream_t s) {
  using A = typename S::A;
  const Geom G = to_geom(a);
  const size_t N = (size_t)a.nx * a.ny;
  if constexpr (is_moments<S>::value) {
    static_assert(MODEL == MODEL_BINARY, "the moment storage holds the binary model");
    if (op == OP_STEP) {
      if (a.bx == 64) return launch_moment<2, S>(a, s);
      if (a.bx == 128) return launch_moment<4, S>(a, s);
      if (a.bx == 256) return launch_moment<8, S>(a, s);
      return cudaErrorInvalidValue;
    }
    // the moment storages keep no populations (g eliminated keeps f and phi)
    if (op == OP_POPS_OUT && pull_kind<S>::value != 2) return cudaErrorNotSupported;
  }
  switch (op) {
    case OP_STEP:
      if constexpr (!is_moments<S>::value) {
        if (a.staged) {
          if ((!is_blocked<S>::value && !staged_fits(a.nx, a.ny)) || !a.err) return cudaErrorInvalidValue;
          if (a.bx == 64) return a.deep ? launch_staged<MODEL, S, 64, 8>(a, s) : launch_staged<MODEL, S, 64, 4>(a, s);
          if (a.bx == 128) return a.deep ? launch_staged<MODEL, S, 128, 6>(a, s) : launch_staged<MODEL, S, 128, 4>(a, s);
          if (a.bx == 256) return a.deep ? launch_staged<MODEL, S, 256, 4>(a, s) : launch_staged<MODEL, S, 256, 3>(a, s);
          return cudaErrorInvalidValue;
        }
        if (a.bx == 64) return launch_step<MODEL, S, 64>(a, s);
        if (a.bx == 128) return launch_step<MODEL, S, 128>(a, s);
        if (a.bx == 256) return launch_step<MODEL, S, 256>(a, s);
      }
      return cudaErrorInvalidValue;
    case OP_INIT:
      init_kernel<MODEL, S><<<grid_for(N, 256), 256, 0, s>>>(G, to_phys<A>(a, MODEL == MODEL_LG), to_buf<S>(a.dst, a), a.in0, a.in1,
                                                              a.in2, a.in3, a.in_cols ? size_t(0) : size_t(a.nx));
      return cudaGetLastError();
    case OP_FIELDS:
      fields_kernel<MODEL, S><<<grid_for(N, 256), 256, 0, s>>>(G, to_buf<S>(a.src, a), a.out0, a.out1, a.out2, a.out3);
      return cudaGetLastError();
    case OP_POPS_OUT:
      if constexpr (!is_moments<S>::value || pull_kind<S>::value == 2)
        pops_out_kernel<MODEL, S><<<grid_for(N, 256), 256, 0, s>>>(G, to_buf<S>(a.src, a), a.flag, a.out0, a.out1);
      return cudaGetLastError();
    case OP_MOMENTS_OUT:
      moments_out_kernel<MODEL, S><<<grid_for(N, 256), 256, 0, s>>>(G, to_buf<S>(a.src, a), a.out0);
      return cudaGetLastError();
    case OP_POPS_IN:
      pops_in_kernel<MODEL, S><<<grid_for(N, 256), 256, 0, s>>>(G, to_buf<S>(a.dst, a), a.in0, a.in1);
      return cudaGetLastError();
    case OP_REDUCE: {
      cudaError_t e = launch_pdl(reduce_partials_kernel<MODEL, S>, a.nparts, RED_THREADS, 0, s, G, to_buf<S>(a.src, a),
                                 a.rho_l, a.rho_g, a.thr, a.partials);
      if (e != cudaSuccess) return e;
      return launch_pdl(reduce_final_kernel<MODEL, S>, 1, RED_FINAL_THREADS, 0, s, G, to_buf<S>(a.src, a), a.thr,
                        a.nparts, (const double*)a.partials, a.red_out, (const int*)a.err);
    }
    case OP_CHECK:
      return read_check_counters(a.check_out);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbk
