// Templated plan: workspace, transform tables, kernel selection and the
// iteration driver, instantiated for float (plan_f32.cu) and double (plan_f64.cu).
#pragma once
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "fft.cuh"
#include "kernel_select.h"
#include "plan_base.h"

namespace dynot {

inline size_t rnd16(size_t b) { return (b + 15) & ~size_t(15); }

// Launch with programmatic dependent launch allowed (the kernels wait for their predecessor with
// griddepcontrol.wait before touching its data; see pdl_wait): the next pass's blocks can be
// scheduled and load their tables while the previous pass drains.  DYNOT_PDL=0 launches plainly.
#ifndef DYNOT_PDL
#define DYNOT_PDL 1
#endif
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = DYNOT_PDL ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

inline size_t tma_smem(int C) {
  switch (C) {
    case 1: return TmaTiles<1>::total;
    case 2: return TmaTiles<2>::total;
    case 3: return TmaTiles<3>::total;
    default: return TmaTiles<4>::total;
  }
}
#ifndef DYNOT_UPD_TMA
#define DYNOT_UPD_TMA 1   // 0: the plain-load update kernel everywhere
#endif

// cuTensorMapEncodeTiled from the driver, resolved once through the runtime
inline PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return (PFN_cuTensorMapEncodeTiled_v12000)f;
  }();
  return fn;
}

template <typename T>
KH<T> pick_kh(int pm) {
  return pm == 16 ? k_hue_t<T, 16> : (pm == 32 ? k_hue_t<T, 32> : k_hue_t<T, 64>);
}

template <typename T>
struct Plan final : PlanBase {
  Geo<T> g{};
  DevMem mem;           // one allocation for every array
  v4<T>* a[2]{};        // a = x - tau sigma K^T bbar, two buffers (current and next)
  v4<T>* b[2]{};        // scaled dual b, two buffers
  T* phi = nullptr;
  T* hat = nullptr;
  v4<T>* x = nullptr;   // primal output x of the last check
  v4<T>* w = nullptr;   // K x0 + (0, f_b^+) at the cells (dual value of a check)
  T* f0n = nullptr;
  T* f1n = nullptr;
  float* stage = nullptr;   // float staging: 2*B*S inputs, then path packing
  size_t stage_floats = 0;
  double* acc = nullptr;    // [B][kAcc]
  double* mass = nullptr;   // [B][P]
  double* chk = nullptr;    // [B][kChk]
  double* scl = nullptr;    // [B][2] densities -> solver units, then [B] solver -> caller units (out_scale)
  double* part = nullptr;   // per-block partial sums of the residual check
  int* err = nullptr;       // set by a kernel whose bounded device wait ran out (sticky until the next start)
  int* active = nullptr;    // [B] per-problem flags of a retiring batch (g.active points here once enabled)
  std::vector<int> h_active;
  // pinned host copies of acc, mass and err, which lie side by side on either side: one copy per check
  double* h_acc = nullptr;
  double* h_mass = nullptr;
  int* h_err = nullptr;
  size_t res_bytes() const { return sizeof(double) * B * kAcc + rnd16(sizeof(double) * (size_t)B * P) + sizeof(int); }
  cudaError_t copy_results() { return cudaMemcpyAsync(h_acc, acc, res_bytes(), cudaMemcpyDeviceToHost, st); }
  // the sums that the per-cell update adds to (the tiled ones write theirs whole)
  cudaError_t clear_results() {
    return tiled ? cudaSuccess : cudaMemsetAsync(acc, 0, sizeof(double) * B * (kAcc + (size_t)P), st);
  }
  // transform tables
  DevMem tabmem;
  XtTables xt{};
  YcTables yc{};
  HueTables ht{};
  int pmax = 32;
  int scrA = 0, scrB = 0;
  size_t smA = 0, smB = 0, smH = 0, smHt = 0;
  KA<T> ka = nullptr;
  KC<T> kc = nullptr;
  bool split_xt = false;    // separate r, x and t launches (the (t, x) plane exceeds shared memory)
  KRX<T> krx_f = nullptr, krx_i = nullptr;
  KCT<T> kct = nullptr;
  int scrS = 0;
  size_t smR = 0, smT = 0;
  KB<T> kb = nullptr;
  size_t smY = 0, smF = 0;
  KFF kff = nullptr;        // FP32, FFT lengths along x: the fused x/t passes
  KFI kfi = nullptr;
  FftXtTables ft{};
  KFY<T> kfy = nullptr;     // FP32, FFT lengths along y: the fused y/colour pass
  KH<T> kh = nullptr;
  // transforms of axes without an FFT length as folded products
  bool x_mm = false, y_mm = false;
  MmAxis<T> mx{}, my{};
  const T *mtf = nullptr, *mti = nullptr;
  KMF<T> kmf = nullptr;
  KMI<T> kmi = nullptr;
  KMY<T> kmy = nullptr;
  size_t smMx = 0, smMi = 0, smMy = 0;
  int ntMf = 0, ntMi = 0, ntMy = 0, wMy = 0;
  // hue transforms as folded products (hue_kernels.cuh); mx holds the bins' tables
  struct HueLaunch {
    int rb = 8, chunk = 0, nch = 1, nt = 0, k = kMmK;   // rows and items per block, blocks per row group, steps per chunk
    size_t smem = 0;
  };
  bool hue_mm = false, hue_small = false;
  HueLaunch hf, hi;
  int hsc = 32;
  size_t smTt = 0;
  const T* htt = nullptr;   // tables of k_hue_tt
  bool tiled = false;       // tiled update kernel (up to four colour channels)
  bool use_tma = false;     // the tiled update stages its planes with bulk tensor copies
  CUtensorMap tmA[2]{}, tmB[2]{}, tmP{};   // a[p], b[p] and phi for k_update_tma
  int tc = 0;               // time-chunk length of the tiled update (autotuned)
  int par = 0;              // buffer holding the current state
  bool have_x = false;
  cudaGraphExec_t gexec[2] = {nullptr, nullptr}, glong[2] = {nullptr, nullptr};   // 2 and kLongGraph iterations
  // [parity][lead]: the check iteration (x written) with its reductions and the copies of the results
  // to pinned host memory, optionally preceded by one plain iteration
  cudaGraphExec_t gcheck[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};
  cudaEvent_t ev[12] = {};

  ~Plan() override {
    for (auto& e : gexec)
      if (e) cudaGraphExecDestroy(e);
    for (auto& e : glong)
      if (e) cudaGraphExecDestroy(e);
    for (auto& row : gcheck)
      for (auto& e : row)
        if (e) cudaGraphExecDestroy(e);
    for (auto& e : ev)
      if (e) cudaEventDestroy(e);
    if (h_acc) cudaFreeHost(h_acc);
  }

  // the FFT paths cover power-of-two axes (DCT for Neumann, real Fourier slots for periodic ones);
  // other lengths take the dense transforms
  bool x_fft() const { return fft_len(n1); }
  bool y_fft() const { return fft_len(n2); }
  size_t xt_smem() const { return xt_layout<T>(nullptr, nullptr, P, n1, pmax, scrA, !x_fft()); }
  size_t yc_smem() const {
    T *t0, *t1, *t2, *t3;
    c2<T> *c0, *c1, *c3;
    return yc_layout<T>(nullptr, C, n2, kW, scrB, !y_fft(), &t0, &c0, &c1, &c3, &t1, &t2, &t3);
  }

  ot_status init() override {
    CUDA_OK(cudaGetDevice(&device));
    pmax = pmax_for(P);
    g.n1 = n1; g.n2 = n2; g.C = C;
    g.per1 = grid.bc[0] == OT_BC_PERIODIC;
    g.per2 = d >= 2 ? grid.bc[1] == OT_BC_PERIODIC : 0;
    g.perc = d >= 3 ? grid.bc[2] == OT_BC_PERIODIC : 0;
    g.P = P; g.S = S; g.B = B; g.N = N;
    g.s1 = (T)grid.axis_scale[0];
    g.s2 = (T)(d >= 2 ? grid.axis_scale[1] : 1.0);
    g.sc = (T)(d >= 3 ? grid.axis_scale[2] : 1.0);
    g.sp = (T)P;
    g.sigma = (T)grid.sigma;
    g.ts = (T)(grid.tau * grid.sigma);

    // ---- workspace
    const size_t cells = (size_t)B * N;
    const size_t narr = 2 * 4 + 2 * 4 + 2 + 4 + 4;
    // staging holds the inputs (2 B S), a packed path (B total) or a packed dual (B (d+1) N)
    stage_floats = std::max<size_t>({2 * (size_t)B * S, (size_t)B * cp.total, (size_t)B * (d + 1) * (size_t)N});
    size_t bytes = narr * rnd16(cells * sizeof(T)) + 2 * rnd16((size_t)B * S * sizeof(T)) +
                   rnd16(stage_floats * sizeof(float)) + rnd16(sizeof(double) * B * kAcc) +
                   rnd16(sizeof(double) * (size_t)B * P) + rnd16(sizeof(double) * B * kChk) +
                   rnd16(sizeof(double) * B * 3) + rnd16(part_bytes()) + 16 + rnd16(sizeof(int) * B);
    CUDA_OK(cudaMalloc(&mem.p, bytes));
    char* q = (char*)mem.p;
    auto take = [&](size_t nb) { char* r = q; q += rnd16(nb); return r; };
    for (int i = 0; i < 2; ++i) a[i] = (v4<T>*)take(cells * sizeof(v4<T>));
    for (int i = 0; i < 2; ++i) b[i] = (v4<T>*)take(cells * sizeof(v4<T>));
    phi = (T*)take(cells * sizeof(T));
    hat = (T*)take(cells * sizeof(T));
    x = (v4<T>*)take(cells * sizeof(v4<T>));
    w = (v4<T>*)take(cells * sizeof(v4<T>));
    f0n = (T*)take((size_t)B * S * sizeof(T));
    f1n = (T*)take((size_t)B * S * sizeof(T));
    stage = (float*)take(stage_floats * sizeof(float));
    acc = (double*)take(sizeof(double) * B * kAcc);
    mass = (double*)take(sizeof(double) * (size_t)B * P);
    err = (int*)take(sizeof(int));
    chk = (double*)take(sizeof(double) * B * kChk);
    scl = (double*)take(sizeof(double) * B * 3);
    part = (double*)take(part_bytes());
    active = (int*)take(sizeof(int) * B);
    CUDA_OK(cudaMemsetAsync(mem.p, 0, bytes, st));

    OT_TRY(build_tables());
    for (auto& e : ev) CUDA_OK(cudaEventCreate(&e));
    CUDA_OK(cudaMallocHost(&h_acc, res_bytes()));
    h_mass = h_acc + (size_t)B * kAcc;
    h_err = (int*)((char*)h_mass + rnd16(sizeof(double) * (size_t)B * P));
    *h_err = 0;
    out_scale.assign(B, 1.0);
    tiled = !hue && C <= 4;
    {
      const char* kind = std::getenv("DYNOT_UPDATE_KERNEL");
      plain_update = kind && std::strcmp(kind, "plain") == 0;
    }
    if constexpr (std::is_same<T, float>::value) {
      // DYNOT_UPDATE_KERNEL=plain selects the plain-load update kernel, =staged the staged one wherever it
      // applies (same arithmetic; for comparisons and profiles)
      const char* kind = std::getenv("DYNOT_UPDATE_KERNEL");
      const bool plain = kind && std::strcmp(kind, "plain") == 0;
      force_staged = kind && std::strcmp(kind, "staged") == 0;
      if (tiled && DYNOT_UPD_TMA && !plain && !g.per1 && !g.per2 && n1 % 4 == 0 && n1 >= kTX && n2 >= kTY)
        OT_TRY(make_tensor_maps());
    }
    OT_TRY(tune());
    {
      // DYNOT_TIME_CHUNK=k: time chunks of k planes in the tiled update instead of the tuned length (comparisons)
      const char* tcs = std::getenv("DYNOT_TIME_CHUNK");
      if (tiled && tcs && std::atoi(tcs) >= 1) tc = std::min(std::atoi(tcs), P);
    }
    return OT_OK;
  }

  // Tensor maps of the TMA-staged update: a and b as float tensors [B P][C][n2][4 n1] (a cell's four components
  // are consecutive, so one box row is one run of 16-byte cells), boxes of 33 x 9 cells (a, with the column left
  // and the row below the 32 x 8 tile) and 32 x 8 cells (b); phi as [B P][C][n2][n1], boxes of 40 x 10 cells.
  // Out-of-range cells read as zero.
  ot_status make_tensor_maps() {
    auto enc = tensor_map_encoder();
    if (!enc) return OT_OK;   // no driver entry point: keep the plain-load update
    const cuuint64_t BP = (cuuint64_t)B * P;
    const cuuint64_t dimS[4] = {4ull * n1, (cuuint64_t)n2, (cuuint64_t)C, BP};
    const cuuint64_t strS[3] = {16ull * n1, 16ull * n1 * n2, 16ull * S};
    const cuuint32_t boxA[4] = {4 * (kTX + 1), kTY + 1, (cuuint32_t)C, 1};
    const cuuint32_t boxB[4] = {4 * kTX, kTY, (cuuint32_t)C, 1};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    for (int i = 0; i < 2; ++i) {
      CUresult r = enc(&tmA[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void*)a[i], dimS, strS, boxA, one,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return OT_OK;   // the driver cannot describe this tensor: keep the plain-load update
      r = enc(&tmB[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void*)b[i], dimS, strS, boxB, one,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return OT_OK;
    }
    const cuuint64_t dim4[4] = {(cuuint64_t)n1, (cuuint64_t)n2, (cuuint64_t)C, BP};
    const cuuint64_t str4[3] = {4ull * n1, 4ull * n1 * n2, 4ull * S};
    const cuuint32_t boxP[4] = {kTX + 8, kTY + 2, (cuuint32_t)C, 1};
    CUresult r = enc(&tmP, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void*)phi, dim4, str4, boxP, one,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return OT_OK;
    const size_t smem = tma_smem(C);
    for (int ck = 0; ck < 2; ++ck)
      for (int wx = 0; wx < 2; ++wx) {
        const void* fn = (const void*)pick_kdt(C, ck, wx);
        CUDA_OK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        // the operands come from shared memory: take the largest shared-memory carve-out of the unified L1
        CUDA_OK(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
      }
    tma_ok = use_tma = true;
    return OT_OK;
  }

  // Autotuner, run once per shape and device (the choice is cached for later plans of the shape):
  //  - the tiled update: staged by bulk tensor copies or with plain loads (where both exist), and time chunks
  //    of P, P/2, P/4 or P/8 planes (3 and 2 on small grids), each timed over whole iterations (FP32).
  // Each candidate is timed over ten launches (after two untimed ones) on the zeroed workspace (b set so that the prox takes its
  // Newton branch); a later candidate must beat the best by 3 % (1 % for the FP32 update, timed over whole iterations,
  // where the update's share dilutes its differences; ties keep the earlier, simpler one).
  struct Tuned {
    int tc = 0;
    bool tma = false;
  };
  static std::mutex& tune_mu() {
    static std::mutex m;
    return m;
  }
  static std::map<std::string, Tuned>& tune_cache() {
    static std::map<std::string, Tuned> c;
    return c;
  }
  std::string shape_key() const {
    char buf[160];
    std::snprintf(buf, sizeof(buf), "%d:%d:%d:%d:%d:%d:%d%d%d:%d:%d%d", (int)sizeof(T), n1, n2, C, P, B, g.per1, g.per2,
                  g.perc, device, (int)tma_ok, (int)force_staged);
    return buf;
  }
  bool tma_ok = false;      // tensor maps exist: the staged update is a candidate
  bool force_staged = false;
  bool plain_update = false;  // DYNOT_UPDATE_KERNEL=plain: no staged kernel, and hue batches update cell by cell

  template <class F>
  ot_status time_launches(F&& launch, float& ms) {
    launch();   // warm
    launch();
    CUDA_OK(cudaGetLastError());
    CUDA_OK(cudaEventRecord(ev[10], st));
    for (int r = 0; r < 10; ++r) launch();
    CUDA_OK(cudaEventRecord(ev[11], st));
    CUDA_OK(cudaEventSynchronize(ev[11]));
    CUDA_OK(cudaEventElapsedTime(&ms, ev[10], ev[11]));
    return OT_OK;
  }

  ot_status tune() {
    std::vector<int> cands;
    for (int d = 1; d <= 8; d *= 2) {
      const int c = (P + d - 1) / d;
      if (c >= 4 || d == 1)
        if (std::find(cands.begin(), cands.end(), c) == cands.end()) cands.push_back(c);
    }
    // small grids: a block's planes follow one another, so shorter chunks on idle SMs pay for the plane they recompute
    if (tiled)
      for (int c : {3, 2}) {
        const dim3 gr = tiled_grid(c);
        if (c < cands.back() && (long long)gr.x * gr.y * gr.z <= 8 * 152) cands.push_back(c);
      }
    tc = cands[0];
    use_tma = tma_ok;
    const std::string key = shape_key();
    {
      std::lock_guard<std::mutex> lk(tune_mu());
      auto it = tune_cache().find(key);
      if (it != tune_cache().end()) {
        tc = it->second.tc;
        use_tma = it->second.tma;
        return OT_OK;
      }
    }
    // a state on which the prox takes its Newton branch: b_f = 1, b_m = 0.5, a = phi = 0
    const long long cells = (long long)B * N;
    k_fill<v4<T>><<<grid1d(cells), 256, 0, st>>>(cells, mk4<T>(T(0.5), T(0.5), T(0.5), T(1)), b[0]);
    CUDA_OK(cudaGetLastError());
    if (tiled) {
      float best = 1e30f;
      Tuned pick{tc, use_tma};
      for (int kind = 0; kind < (tma_ok && !force_staged ? 2 : 1); ++kind) {
        use_tma = tma_ok && kind == 0;
        for (int c : cands) {
          tc = c;
          float ms = 0;
          // FP32: whole iterations, the update's time with phi just written by the inverse pass, as in a solve
          // (timed alone, on a cold workspace, the ranking of the time chunks differed from the one inside
          // iterations); FP64 (the precision study's reference, whose iterations are long): the update alone
          if (std::is_same<T, float>::value) OT_TRY(time_launches([&] { enqueue_iteration(0, false, false); }, ms));
          else OT_TRY(time_launches([&] { enqueue_update(0, false, false); }, ms));
          if (ms < (std::is_same<T, float>::value ? 0.99f : 0.97f) * best) {   // whole iterations: 1 %
            best = ms;
            pick.tc = c;
            pick.tma = use_tma;
          }
        }
      }
      tc = pick.tc;
      use_tma = pick.tma;
    }
    tune_tc = tc;
    // clear both buffer sets again
    for (int i = 0; i < 2; ++i) {
      CUDA_OK(cudaMemsetAsync(a[i], 0, (size_t)B * N * sizeof(v4<T>), st));
      CUDA_OK(cudaMemsetAsync(b[i], 0, (size_t)B * N * sizeof(v4<T>), st));
    }
    std::lock_guard<std::mutex> lk(tune_mu());
    tune_cache()[key] = Tuned{tc, use_tma};
    return OT_OK;
  }
  int tune_tc = 0;

  static MmAxis<T> mm_shape(int n, bool per) {
    MmAxis<T> ax{};
    ax.n = n;
    ax.h0 = per ? n / 2 + 1 : (n + 1) / 2;
    ax.h1 = n - ax.h0;
    ax.o1 = per;
    ax.l0 = ax.li = (ax.h0 + 3) / 4 * 4;
    ax.lf = ax.l0 + (ax.h1 + 3) / 4 * 4;
    return ax;
  }

  // Multiply-adds of the FP64 pipe on the busiest quarter of an SM, in warp instructions: `blocks` blocks of `warps`
  // warps, `steps` instructions each.  The pipe takes a warp's instruction in the same time whatever its active lanes.
  static long long fp64_load(long long blocks, long long warps, long long steps) {
    constexpr int sms = 152, quarters = 4;
    return ((blocks + sms - 1) / sms * warps + quarters - 1) / quarters * steps;
  }
  static long long warps_of(long long items) { return (items + 31) / 32; }

  // The hue transforms as folded products, where the rows fit shared memory (at 16 rows per block and P > 8 up to 2339
  // bins in FP32; not every length below the last that fits: the chunks of an axis differ).
  //  - Few row groups (a single pair): the latency-bound form of the kernels, where its table columns fit and, in FP32,
  //    its blocks, which form their 8 rows' r again for every 16 items, run in at most four waves (720 bins, P = 32:
  //    8 pairs in 3 waves 61 us an iteration against 71, 16 pairs in 6 waves 101 against 82).
  //  - FP32: 16 rows per block and the fewest chunks of items, the least table traffic, where these blocks fill the GPU;
  //    as many chunks as two blocks per SM hold where they would leave some SMs with two blocks and some with one
  //    (850 bins, P = 40, 32 pairs 196 -> 174 us).  Fewer blocks: 8 rows, and chunks (of a warp's lanes at least) up to
  //    one block per SM (720 bins, 16 pairs 101 -> 82 us; 1000 bins, P = 64, 8 pairs 140 -> 120).
  //  - FP32: steps in chunks of 16, which wait half as often for copies, unless fewer blocks would share an SM
  //    (1000 bins, P = 64, 64 pairs 640 -> 593 us; 500 bins, 64 pairs would take 192 instead of 173).
  //  - FP64: the per-row kernels where they load the FP64 pipe less (720 bins, P = 32, one pair 1331 -> 326 us;
  //    180 bins, P = 36, 32 pairs 366 -> 345; 360 bins, P = 64, one pair keeps the products, 95 against 133).
  ot_status choose_hue_mm() {
    int maxsm = 0, smsm = 0, reserved = 0;
    CUDA_OK(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
    CUDA_OK(cudaDeviceGetAttribute(&smsm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device));
    CUDA_OK(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, device));
    constexpr bool fp64 = sizeof(T) == 8;
    constexpr int sms = 152;
    mx = mm_shape(n1, true);
    const int items_f = mx.lf / 4, items_i = (mx.h0 + 1) / 2;   // outputs per 8 rows, 4 table columns each
    const long long G8 = (long long)((P + 7) / 8) * B, G16 = (long long)((P + 15) / 16) * B;
    const size_t smem_small = sizeof(T) * hue_mm_vals(n1, mx.h0, 8, kHueItems, true);
    auto resident = [&](size_t smem, int nt) {   // blocks per SM, at 128 registers
      return std::max<long long>(1, std::min<long long>(smsm / ((long long)smem + reserved), 65536 / (128 * nt)));
    };
    auto waves = [&](int items) {
      const long long per = sms * resident(smem_small, kHueMmThreads);
      return (G8 * ((items + kHueItems - 1) / kHueItems) + per - 1) / per;
    };
    hue_small = G8 < sms && (int)smem_small <= maxsm && (fp64 || std::max(waves(items_f), waves(items_i)) <= 4);
    auto pick = [&](int items, int even) {
      HueLaunch h;
      if (hue_small) {
        h.chunk = kHueItems;
        h.nt = kHueMmThreads;
        h.nch = (items + h.chunk - 1) / h.chunk;
        h.smem = smem_small;
        return h;
      }
      auto least = [&](int rb) { return (items + kHueMmThreads / (rb / 8) - 1) / (kHueMmThreads / (rb / 8)); };
      h.rb = P > 8 ? 16 : 8;
      h.nch = least(h.rb);
      if (!fp64) {
        if (P > 8 && G16 * h.nch < 92) h.rb = 8;
        if (h.rb == 8) {
          h.nch = std::max<int>(least(8), (int)std::min<long long>(sms / G8, items / 32));
        } else if (G16 * h.nch > sms) {
          h.nch = std::max<int>(h.nch, (int)(2 * sms / G16));
        }
      }
      h.chunk = ((items + h.nch - 1) / h.nch + even - 1) / even * even;
      h.nch = (items + h.chunk - 1) / h.chunk;
      h.nt = std::max(128, (h.rb / 8 * h.chunk + 31) / 32 * 32);
      h.smem = sizeof(T) * hue_mm_vals(n1, mx.h0, h.rb, h.chunk, false);
      if (!fp64) {
        const size_t s16 = sizeof(T) * hue_mm_vals(n1, mx.h0, h.rb, h.chunk, false, 16);
        const long long per_sm = ((h.rb == 8 ? G8 : G16) * h.nch + sms - 1) / sms;
        if ((int)s16 <= maxsm && resident(s16, h.nt) >= std::min(per_sm, resident(h.smem, h.nt))) {
          h.k = 16;
          h.smem = s16;
        }
      }
      return h;
    };
    hf = pick(items_f, 1);
    hi = pick(items_i, 2);
    hsc = hue_small ? HueTt<true>::SC : HueTt<false>::SC;
    smTt = sizeof(T) * hue_tt_vals(P, hsc);
    hue_mm = (int)std::max(std::max(hf.smem, hi.smem), smTt) <= maxsm && hf.nt <= kHueMmThreads && hi.nt <= kHueMmThreads;
    if (fp64 && hue_mm) {
      // both bin transforms and the time transforms (P^2 or, per row, 2 P pmax multiply-adds per slot)
      const long long hpad = hue_hpad(mx.h0), cols = (long long)n1 * B * P / (32 * 4 * sms);
      auto load = [&](const HueLaunch& h) {
        return hue_small ? fp64_load(G8 * h.nch, kHueMmThreads / 32, 32 * hpad / kHueSlices)
                         : fp64_load((long long)((P + h.rb - 1) / h.rb) * B * h.nch, warps_of(h.rb / 8 * h.chunk), 32 * hpad);
      };
      hue_mm = load(hf) + load(hi) + cols * P <= 1.05 * (fp64_load((long long)P * B, warps_of(n1), 2ll * n1) + cols * 2 * pmax);
    }
    return OT_OK;
  }

  // Axes without an FFT length take the folded products where a (x, t) plane (x) or a strip of columns (y) fits
  // shared memory and a strip's outputs fit one block's registers; the dense sums keep the rest.  In FP32 that is x axes
  // beyond 1093 cells (P = 9), 760 (P = 24), 624 (P = 32), 458 (P = 48) or 359 (P = 64) and y axes beyond 1024; in FP64
  // half of that or less.  The FP64 plan also keeps the dense sums where they load the pipe less: the products halve the
  // multiply-adds, but a thread holds 32 to 48 sums, and short axes leave most of an SM's quarters without a warp.
  ot_status choose_mm() {
    int maxsm = 0;
    CUDA_OK(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
    const char* sx = std::getenv("DYNOT_SPLIT_XT");
    const bool split = sx && std::strcmp(sx, "1") == 0;
    mx = mm_shape(n1, g.per1);
    my = mm_shape(n2, g.per2);
    constexpr bool fp64 = sizeof(T) == 8;
    auto lanes = [](int items) { return items / (32.0 * ((items + 31) / 32)); };
    const int bufx = mm_buf(mx.l0, mx.lf, mx.li), bufy = mm_buf(my.l0, my.lf, my.li);
    auto round = [](int n, int lo, int hi) { return std::max(lo, std::min(hi, (n + 31) / 32 * 32)); };
    if (!x_fft() && !split) {
      const int pm = mm_pm(P), dense = 4 * n1, G = (P + 7) / 8;
      const size_t old = xt_layout<T>(nullptr, nullptr, P, n1, pmax, dense, true);
      smMx = mm_xt_smem<T>(n1, P, pm, bufx, true);
      smMi = mm_xt_smem<T>(n1, P, pm, bufx, false);
      // Both passes, the time transforms included.  Measured (us, forward and inverse pass, dense | products): 63, P = 9
      // 52 | 97; 33x2x3, P = 12 46 | 64; 150x24x3, P = 12 182 | 212; 40x48x3, P = 32 146 | 114; 110x66x3, P = 64 1430 |
      // 785.  400 instructions (13 us) are what the products' barriers and table copies cost beside them.
      const long long nb = (long long)n2 * C * B, cols = warps_of(n1), P4 = (P + 3) / 4 * 4, hP4 = ((P + 1) / 2 + 3) / 4 * 4;
      const bool less = fp64_load(nb, cols, P4 * pm / 2 + hP4 * pm) + fp64_load(nb, warps_of(G * (mx.lf / 4)), 32ll * mx.h0) +
                            fp64_load(nb, warps_of(G * ((mx.h0 + 1) / 2)), 32ll * mx.h0) + 400 <
                        fp64_load(nb, cols, 2ll * P * pmax) + fp64_load(nb, 8 * ((P * n1 + 255) / 256), 2ll * n1);
      // (the kernels' offsets into a problem's a are 32-bit)
      if ((int)smMx <= maxsm && (int)old <= maxsm && 4 * N < (1ll << 31) && (!fp64 || less)) {
        x_mm = true;
        kmf = pick_kmf<T>(pm);
        kmi = pick_kmi<T>(pm);
        // threads: the products' items in equal rounds, up to 160 (three or four blocks per SM) where the grid fills the
        // GPU and as many as have work otherwise
        const int most = nb > 2 * 152 ? 160 : kMmXtThreads;
        const int work = G * (mx.lf / 4), rounds = (work + most - 1) / most;
        ntMf = ntMi = round(std::max((work + rounds - 1) / rounds, std::min(n1, 96)), 64, most);
      }
    }
    if (!y_fft()) {
      const int wt = mm_yc_wt(C);
      // FP64: the load of the dense sums (strips of kW columns, both transforms) less what the products' folding, barriers
      // and copies cost beside them, about 200 instructions and a twentieth.  Measured (us, dense | products):
      // 32x30x3, P = 9 27 | 75; 128x40x3, P = 16 65 | 96; 40x48x3, P = 32 80 | 100; 64x150x1, P = 16 111 | 193;
      // 128x75x3, P = 24 253 | 225; 58x59x3, P = 48 166 | 146; 143x160x3, P = 40 1637 | 1181; 36x160x3, P = 25 342 | 399
      // with strips of 16 columns, 305 with 8.  Between strips of the same load the share of lanes and columns at work
      // decides (100x100x1, P = 32 141 us with 16 columns, 133 with 8).
      double load = fp64_load((long long)((n1 + kW - 1) / kW) * P * B, 8 * ((kW * C * n2 + 255) / 256), 2ll * n2) / 0.95 - 200;
      double best = 0;
      for (int w = 16; w >= wt; w /= 2) {
        const int items = mm_yc_items(my.lf, C, w);
        const size_t sm = mm_yc_smem<T>(n2, C, w, bufy);
        if (fp64) {
          const long long nb = (long long)((n1 + w - 1) / w) * P * B, steps = 4ll * wt * C * my.h0;
          const double l = (double)(fp64_load(nb, warps_of(items), steps) + fp64_load(nb, warps_of(w / wt * ((my.h0 + 1) / 2)), steps));
          const double use = lanes(items) * n1 / ((n1 + w - 1) / w * w);
          if (items > kMmYcThreads || (int)sm > maxsm || l > load || (l == load && use <= best)) continue;
          load = l;
          best = use;
          y_mm = true;
          wMy = w;
          smMy = sm;
          kmy = pick_kmy<T>(C);
          ntMy = round(items, 64, kMmYcThreads);
          continue;
        }
        // narrower strips while the grid has fewer than three blocks per SM (180x135x3x24: 40.0 us with 8 columns, 42.5
        // with 16; 300x200x3x16: 63.2 against 67.2)
        const bool more = w > wt && (long long)((n1 + w - 1) / w) * P * B < 3 * 152;
        if (items > kMmYcThreads || (int)sm > maxsm || more) continue;
        y_mm = true;
        wMy = w;
        smMy = sm;
        kmy = pick_kmy<T>(C);
        ntMy = round(items, 128, kMmYcThreads);
        break;
      }
    }
    return OT_OK;
  }

  // ---- transform tables (computed in double on the host)
  ot_status build_tables() {
    std::vector<char> h;
    // tables start on whole lines: a warp's copy of 512 bytes is then four of them (333 bins, P = 27, 32 pairs: the time
    // transforms 16.6 us from a table that starts between them, 11.8 like this)
    auto line = [](size_t nb) { return (nb + 255) / 256 * 256; };
    auto put = [&](const void* src, size_t nb) {
      size_t off = h.size();
      h.resize(off + line(nb));
      std::memcpy(h.data() + off, src, nb);
      return off;
    };
    auto twid = [&](int n, std::vector<T>& tw, std::vector<T>& hw) {
      tw.resize(2 * n);
      hw.resize(2 * n);
      for (int j = 0; j < n; ++j) {
        tw[2 * j] = (T)std::cos(2 * kPi * j / n);
        tw[2 * j + 1] = (T)-std::sin(2 * kPi * j / n);
        hw[2 * j] = (T)std::cos(kPi * j / (2.0 * n));
        hw[2 * j + 1] = (T)-std::sin(kPi * j / (2.0 * n));
      }
    };
    auto cos4 = [&](int n) {
      std::vector<T> c(4 * n);
      for (int m = 0; m < 4 * n; ++m) c[m] = (T)std::cos(kPi * m / (2.0 * n));
      return c;
    };
    auto neu_lam = [&](int n, double s) {
      std::vector<double> l(n);
      for (int j = 0; j < n; ++j) {
        const double v = std::sin(kPi * j / (2.0 * n));
        l[j] = s * s * 4.0 * v * v;
      }
      return l;
    };
    // periodic axis: eigenvalue of each real-Fourier slot (rdft_dense_rows), frequency (slot + 1) / 2
    auto per_lam = [&](int n, double s) {
      std::vector<double> l(n);
      for (int slot = 0; slot < n; ++slot) {
        const int j = (n % 2 == 0 && slot == n - 1) ? n / 2 : (slot + 1) / 2;
        const double v = std::sin(kPi * j / n);
        l[slot] = s * s * 4.0 * v * v;
      }
      return l;
    };
    // an axis transformed by folded products: its spectrum order [even part][odd part], eigenvalues in that order
    auto mm_freq = [](int n, bool per, int pos) {   // frequency at a position of the spectrum
      const int h0 = per ? n / 2 + 1 : (n + 1) / 2;
      return per ? (pos < h0 ? pos : pos - h0 + 1) : (pos < h0 ? 2 * pos : 2 * (pos - h0) + 1);
    };
    auto mm_lam = [&](int n, bool per, double s) {
      std::vector<double> l(n);
      for (int q = 0; q < n; ++q) {
        const double v = std::sin(kPi * mm_freq(n, per, q) / (per ? n : 2.0 * n));
        l[q] = s * s * 4.0 * v * v;
      }
      return l;
    };
    // Its tables, zero up to whole groups of 16 rows (read by the hue kernels), are filled on the device (k_mm_tables) behind
    // the host's; off: turn, turn2, then ft and it from the end of the host's tables.
    size_t dev = 0;
    auto mm_axis = [&](const MmAxis<T>& ax, size_t (&off)[4]) {
      const int n = ax.n;
      std::vector<T> turn(4 * n), turn2(4 * n);
      for (int m = 0; m < 4 * n; ++m) {
        const double v = std::cos(2 * kPi * m / (4.0 * n));
        turn[m] = (T)v;
        turn2[m] = (T)(2.0 / n * v);
      }
      off[0] = put(turn.data(), turn.size() * sizeof(T));
      off[1] = put(turn2.data(), turn2.size() * sizeof(T));
      const size_t rows = hue_hpad(ax.h0);
      off[2] = dev;
      dev += line(rows * ax.lf * sizeof(T));
      off[3] = dev;
      dev += line(rows * 2 * ax.li * sizeof(T));
    };
    size_t o_mx[4] = {}, o_my[4] = {}, o_mtf = 0, o_mti = 0;
    // (cos, sin)(2 pi m / n) pairs, padded to the 4 n values of the cosine table they replace
    auto cs_pad = [&](int n) {
      std::vector<T> c(4 * n, T(0));
      for (int m = 0; m < n; ++m) {
        c[2 * m] = (T)std::cos(2 * kPi * m / n);
        c[2 * m + 1] = (T)std::sin(2 * kPi * m / n);
      }
      return c;
    };
    auto toT = [&](const std::vector<double>& v) {
      std::vector<T> r(v.size());
      for (size_t i = 0; i < v.size(); ++i) r[i] = (T)v[i];
      return r;
    };
    // cos(pi m / 2P), for the folded time transforms
    std::vector<double> cosP(4 * P);
    for (int m = 0; m < 4 * P; ++m) cosP[m] = std::cos(kPi * (double)m / (2.0 * P));
    // time axis: forward and inverse DCT matrices, padded to pmax columns
    std::vector<T> Mf((size_t)P * pmax, T(0)), Mi((size_t)P * pmax, T(0));
    for (int k = 0; k < P; ++k)
      for (int t = 0; t < P; ++t) {
        const double c = std::cos(kPi * k * (2 * t + 1) / (2.0 * P));
        Mf[(size_t)k * pmax + t] = (T)c;
        Mi[(size_t)t * pmax + k] = (T)((k == 0 ? 1.0 : 2.0) / P * c);
      }
    const std::vector<double> lt = neu_lam(P, (double)P);
    const double thr = grid.precision == OT_PREC_MIXED ? grid.lam_fp64 : 0.0;

    std::vector<T> twt(2 * P), hwt(2 * P);
    for (int j = 0; j < P; ++j) {
      twt[2 * j] = (T)std::cos(2 * kPi * j / P);
      twt[2 * j + 1] = (T)-std::sin(2 * kPi * j / P);
      hwt[2 * j] = (T)std::cos(kPi * j / (2.0 * P));
      hwt[2 * j + 1] = (T)-std::sin(kPi * j / (2.0 * P));
    }
    size_t o_twt = put(twt.data(), twt.size() * sizeof(T));
    size_t o_hwt = put(hwt.data(), hwt.size() * sizeof(T));
    size_t o_Mf = put(Mf.data(), Mf.size() * sizeof(T));
    size_t o_Mi = put(Mi.data(), Mi.size() * sizeof(T));
    std::vector<T> ltT = toT(lt);
    size_t o_lt = put(ltT.data(), P * sizeof(T));
    size_t o_ltd = put(lt.data(), P * sizeof(double));

    size_t o_tw1 = 0, o_hw1 = 0, o_c41 = 0, o_tw2 = 0, o_hw2 = 0, o_c42 = 0, o_l1 = 0, o_l1d = 0, o_l2 = 0,
           o_l2d = 0, o_Q = 0, o_lc = 0, o_lcd = 0, o_cs = 0, o_hl = 0, o_hld = 0, o_tt = 0;
    if (!hue) {
      std::vector<T> tw, hw;
      twid(n1, tw, hw);
      o_tw1 = put(tw.data(), tw.size() * sizeof(T));
      o_hw1 = put(hw.data(), hw.size() * sizeof(T));
      std::vector<T> c1 = g.per1 ? cs_pad(n1) : cos4(n1);
      o_c41 = put(c1.data(), c1.size() * sizeof(T));
      twid(n2, tw, hw);
      o_tw2 = put(tw.data(), tw.size() * sizeof(T));
      o_hw2 = put(hw.data(), hw.size() * sizeof(T));
      std::vector<T> c2v = g.per2 ? cs_pad(n2) : cos4(n2);
      o_c42 = put(c2v.data(), c2v.size() * sizeof(T));
      OT_TRY(choose_mm());
      if (x_mm) mm_axis(mx, o_mx);
      if (x_mm || (x_fft() && P < pmax)) {   // folded time transforms
        const int pm = x_mm ? mm_pm(P) : pmax, ph = pm / 2, hP = (P + 1) / 2, P4 = (P + 3) / 4 * 4, hP4 = (hP + 3) / 4 * 4;
        std::vector<T> tf((size_t)P4 * ph, T(0)), ti((size_t)hP4 * pm, T(0));
        for (int k = 0; k < P; ++k)
          for (int t = 0; t < P; ++t) {
            const double c = cosP[k * (2 * t + 1) % (4 * P)];
            if (t < hP) tf[(size_t)k * ph + t] = (T)c;
            if (t < hP4) ti[(size_t)t * pm + (k & 1) * ph + k / 2] = (T)((k == 0 ? 1.0 : 2.0) / P * c);
          }
        o_mtf = put(tf.data(), tf.size() * sizeof(T));
        o_mti = put(ti.data(), ti.size() * sizeof(T));
      }
      if (y_mm) mm_axis(my, o_my);
      const double s2y = d >= 2 ? grid.axis_scale[1] : 1.0;
      std::vector<double> l1 = x_mm ? mm_lam(n1, g.per1, grid.axis_scale[0])
                                    : (g.per1 ? per_lam(n1, grid.axis_scale[0]) : neu_lam(n1, grid.axis_scale[0]));
      std::vector<double> l2 = y_mm ? mm_lam(n2, g.per2, s2y) : (g.per2 ? per_lam(n2, s2y) : neu_lam(n2, s2y));
      std::vector<T> l1T = toT(l1), l2T = toT(l2);
      o_l1 = put(l1T.data(), n1 * sizeof(T));
      o_l1d = put(l1.data(), n1 * sizeof(double));
      o_l2 = put(l2T.data(), n2 * sizeof(T));
      o_l2d = put(l2.data(), n2 * sizeof(double));
      // colour axis: orthonormal eigenbasis of its 1D Laplacian
      std::vector<double> Q((size_t)C * C, 0.0), lc(C, 0.0);
      const double sc = d >= 3 ? grid.axis_scale[2] : 1.0;
      if (!g.perc) {  // Neumann: DCT-II basis, eigenvalues 4 sin^2(pi j / 2C)
        for (int j = 0; j < C; ++j) {
          const double v = std::sin(kPi * j / (2.0 * C));
          lc[j] = sc * sc * 4 * v * v;
          for (int c = 0; c < C; ++c)
            Q[(size_t)c * C + j] = std::sqrt((j == 0 ? 1.0 : 2.0) / C) * std::cos(kPi * j * (2 * c + 1) / (2.0 * C));
        }
      } else {        // periodic: real Fourier basis, eigenvalues 4 sin^2(pi f / C)
        for (int j = 0; j < C; ++j) {
          const int f = (j + 1) / 2;
          const double v = std::sin(kPi * f / C);
          lc[j] = sc * sc * 4 * v * v;
          for (int c = 0; c < C; ++c) {
            double q;
            if (j == 0) q = 1.0 / std::sqrt((double)C);
            else if (C % 2 == 0 && j == C - 1) q = ((c & 1) ? -1.0 : 1.0) / std::sqrt((double)C);
            else if (j & 1) q = std::sqrt(2.0 / C) * std::cos(2 * kPi * f * c / C);
            else q = std::sqrt(2.0 / C) * std::sin(2 * kPi * f * c / C);
            Q[(size_t)c * C + j] = q;
          }
        }
      }
      std::vector<T> QT = toT(Q), lcT = toT(lc);
      o_Q = put(QT.data(), QT.size() * sizeof(T));
      o_lc = put(lcT.data(), C * sizeof(T));
      o_lcd = put(lc.data(), C * sizeof(double));
    } else {
      const int n = n1;
      std::vector<T> cs(2 * n);
      OT_TRY(choose_hue_mm());
      if (hue_mm) {
        mm_axis(mx, o_mx);
        const int hP = (P + 1) / 2, P4 = hue_p4(P), h4 = hue_h4(P);
        std::vector<T> tt((size_t)hP * P4 + 2 * (size_t)hP * h4, T(0));
        T *te = tt.data() + (size_t)hP * P4, *to = te + (size_t)hP * h4;
        for (int k = 0; k < P; ++k)
          for (int t = 0; t < hP; ++t) {
            const double c = cosP[k * (2 * t + 1) % (4 * P)];
            tt[(size_t)t * P4 + k] = (T)c;
            (k & 1 ? to : te)[(size_t)(k / 2) * h4 + t] = (T)((k == 0 ? 1.0 : 2.0) / P * c);
          }
        o_tt = put(tt.data(), tt.size() * sizeof(T));
      }
      std::vector<double> hl(n);
      for (int m = 0; m < n; ++m) {
        cs[2 * m] = (T)std::cos(2 * kPi * m / n);
        cs[2 * m + 1] = (T)std::sin(2 * kPi * m / n);
      }
      hl = hue_mm ? mm_lam(n, true, grid.axis_scale[0]) : per_lam(n, grid.axis_scale[0]);
      std::vector<T> hlT = toT(hl);
      o_cs = put(cs.data(), cs.size() * sizeof(T));
      o_hl = put(hlT.data(), n * sizeof(T));
      o_hld = put(hl.data(), n * sizeof(double));
    }
    CUDA_OK(cudaMalloc(&tabmem.p, h.size() + dev));
    CUDA_OK(cudaMemcpyAsync(tabmem.p, h.data(), h.size(), cudaMemcpyHostToDevice, st));
    char* base = (char*)tabmem.p;
    auto mm_fill = [&](MmAxis<T>& ax, const size_t (&off)[4]) -> ot_status {
      T *ft = (T*)(base + h.size() + off[2]), *it = (T*)(base + h.size() + off[3]);
      ax.ft = ft;
      ax.it = it;
      k_mm_tables<T><<<dim3((ax.lf + 2 * ax.li + 127) / 128, hue_hpad(ax.h0)), 128, 0, st>>>(
          ax, (const T*)(base + off[0]), (const T*)(base + off[1]), ft, it);
      CUDA_OK(cudaGetLastError());
      return OT_OK;
    };
    if (!hue) {
      xt.tw = base + o_tw1; xt.hw = base + o_hw1; xt.cos4 = base + o_c41;
      xt.Mt_f = base + o_Mf; xt.Mt_i = base + o_Mi;
      xt.twt = base + o_twt; xt.hwt = base + o_hwt;
      yc.tw = base + o_tw2; yc.hw = base + o_hw2; yc.cos4 = base + o_c42;
      yc.lam1 = base + o_l1; yc.lam2 = base + o_l2; yc.lamt = base + o_lt;
      yc.lam1d = (const double*)(base + o_l1d); yc.lam2d = (const double*)(base + o_l2d);
      yc.lamtd = (const double*)(base + o_ltd);
      yc.Qc = base + o_Q; yc.lamc = base + o_lc; yc.lamcd = (const double*)(base + o_lcd);
      yc.lam_fp64 = thr;
      if (x_mm) OT_TRY(mm_fill(mx, o_mx));
      xt.late = sizeof(T) == 8 && !(x_fft() && y_fft());
      mtf = (const T*)(base + o_mtf);
      mti = (const T*)(base + o_mti);
      if (y_mm) OT_TRY(mm_fill(my, o_my));
      scrA = x_fft() ? (kThreadsXt / fft_n1(n1)) * n1 : 4 * n1;
      scrB = y_fft() ? (yc_threads(n2) / fft_n1(n2)) * n2 : 4 * n2;
      ka = pick_ka<T>(x_fft() ? n1 : 0, pmax);
      kc = pick_kc<T>(x_fft() ? n1 : 0, pmax);
      kb = pick_kb<T>(y_fft() ? n2 : 0);
      if constexpr (std::is_same<T, float>::value) kfy = y_fft() ? pick_kfy<T>(n2, C) : nullptr;
      if (kfy) smY = fft_yc_smem<T>(fft_n1(n2), n2 / fft_n1(n2), C);
      smA = xt_smem();
      smB = yc_smem();
      int maxsm = 0;
      CUDA_OK(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
      // a (t, x) plane too large for one block's shared memory takes the split x/t passes
      // (DYNOT_SPLIT_XT=1 selects them for any grid, for comparisons)
      const char* sx = std::getenv("DYNOT_SPLIT_XT");
      split_xt = !x_mm && ((int)smA > maxsm || (sx && std::strcmp(sx, "1") == 0));
      if (split_xt) {
        scrS = x_fft() ? (256 / fft_n1(n1)) * n1 : (kRowsX * n1 + 1) / 2;
        T *t0p, *t1p;
        c2<T> *c0p, *c1p, *c2p;
        smR = rows_x_layout<T>(nullptr, n1, scrS, !x_fft(), &t0p, &c0p, &c1p, &c2p, &t1p);
        smT = sizeof(T) * ((size_t)P * pmax + (size_t)P * kColsT);
        krx_f = pick_krx<T, false>(x_fft() ? n1 : 0);
        krx_i = pick_krx<T, true>(x_fft() ? n1 : 0);
        kct = pick_kct<T>(pmax);
      }
      if constexpr (std::is_same<T, float>::value) {
        if (x_fft() && !split_xt) {
          kff = pick_kff(n1, pmax);
          kfi = pick_kfi(n1, pmax);
          smF = fft_xt_smem(n1, P, pmax);
          ft = FftXtTables{(const float2*)xt.tw, (const float2*)xt.hw, (const float2*)xt.twt, (const float2*)xt.hwt, mtf, mti};
          CUDA_OK(cudaFuncSetAttribute((const void*)kff, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
          CUDA_OK(cudaFuncSetAttribute((const void*)kfi, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
        }
      }
      if ((!split_xt && (int)smA > maxsm) || (int)smB > maxsm || (split_xt && ((int)smR > maxsm || (int)smT > maxsm)))
        return seterr(OT_EUNSUPPORTED, "grid needs %zu / %zu bytes of shared memory per block (max %d)",
                      split_xt ? std::max(smR, smT) : smA, smB, maxsm);
      // The limit is a property of the kernel, shared by every plan that uses it:
      // raise it to the device maximum instead of this plan's size.
      if (split_xt) {
        CUDA_OK(cudaFuncSetAttribute((const void*)krx_f, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
        CUDA_OK(cudaFuncSetAttribute((const void*)krx_i, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
        CUDA_OK(cudaFuncSetAttribute((const void*)kct, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
      } else {
        CUDA_OK(cudaFuncSetAttribute((const void*)ka, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
        CUDA_OK(cudaFuncSetAttribute((const void*)kc, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
      }
      CUDA_OK(cudaFuncSetAttribute((const void*)kb, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
      for (const void* f : {(const void*)kmf, (const void*)kmi, (const void*)kmy, (const void*)kfy})
        if (f) CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
    } else {
      ht.cs = base + o_cs; ht.lam = base + o_hl; ht.lamd = (const double*)(base + o_hld);
      ht.lamt = base + o_lt; ht.lamtd = (const double*)(base + o_ltd);
      ht.Mt_f = base + o_Mf; ht.Mt_i = base + o_Mi;
      ht.lam_fp64 = thr;
      kh = pick_kh<T>(pmax);
      smH = rnd16(sizeof(T) * n1) + rnd16(sizeof(c2<T>) * n1);
      smHt = hue_t_smem_for<T>(pmax);
      int maxsm = 0;
      CUDA_OK(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
      if ((int)smH > maxsm || (int)smHt > maxsm)
        return seterr(OT_EUNSUPPORTED, "hue grid needs %zu / %zu bytes of shared memory per block (max %d)", smH,
                      smHt, maxsm);
      CUDA_OK(cudaFuncSetAttribute((const void*)k_hue_fwd<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
      CUDA_OK(cudaFuncSetAttribute((const void*)k_hue_inv<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
      CUDA_OK(cudaFuncSetAttribute((const void*)kh, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
      if (hue_mm) {
        OT_TRY(mm_fill(mx, o_mx));
        htt = (const T*)(base + o_tt);
        if constexpr (sizeof(T) == 4)
          for (const void* f : {(const void*)k_hue_x_fwd<T, false, 16>, (const void*)k_hue_x_inv<T, false, 16>})
            CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
        for (const void* f : {(const void*)k_hue_x_fwd<T, true, kMmK>, (const void*)k_hue_x_fwd<T, false, kMmK>,
                              (const void*)k_hue_x_inv<T, true, kMmK>, (const void*)k_hue_x_inv<T, false, kMmK>,
                              (const void*)k_hue_tt<T, true>, (const void*)k_hue_tt<T, false>})
          CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
      }
    }
    return OT_OK;
  }

  Arrays<T> arrays(int p, bool wx) const {
    Arrays<T> A{};
    A.a = a[p];
    A.b = b[p];
    A.an = a[1 - p];
    A.bn = b[1 - p];
    A.x = wx ? x : nullptr;
    A.w = w;
    A.phi = phi;
    A.f0 = f0n;
    A.f1 = f1n;
    return A;
  }
  const v4<T>* aptr(int p) const { return a[p]; }

  // ---- the Poisson solve phi = (A A^T)^+ (A a - f_b^-) for a in buffer p
  void enqueue_poisson(int p, cudaEvent_t* evs) { enqueue_poisson_src(aptr(p), evs); }
  void enqueue_poisson_src(const v4<T>* asrc, cudaEvent_t* evs) {
    if (!hue) {
      if (evs) cudaEventRecord(evs[0], st);
      bool done = false;
      if constexpr (std::is_same<T, float>::value) {
        if (kff) {
          launch_pdl(kff, dim3(C, n2, B), dim3(fft_xt_threads(n1, pmax)), smF, st, g, asrc, (const T*)f0n, (const T*)f1n,
                     hat, ft);
          done = true;
        }
      }
      if (done) {
      } else if (x_mm) {
        launch_pdl(kmf, dim3(C, n2, B), dim3(ntMf), smMx, st, g, asrc, (const T*)f0n, (const T*)f1n, hat, mx, mtf);
      } else if (split_xt) {
        k_rhs_cells<T><<<grid1d((long long)B * N), 256, 0, st>>>(g, asrc, (const T*)f0n, (const T*)f1n, hat);
        launch_pdl(krx_f, dim3((P + kRowsX - 1) / kRowsX, n2 * C, B), dim3(256), smR, st, g, (const T*)hat, hat, xt,
                   scrS);
        launch_pdl(kct, dim3((n1 + kColsT - 1) / kColsT, n2 * C, B), dim3(kColsT), smT, st, g, hat,
                   (const T*)xt.Mt_f);
      } else {
        launch_pdl(ka, dim3(n2, C, B), dim3(kThreadsXt), smA, st, g, asrc, (const T*)f0n, (const T*)f1n, hat, xt,
                   scrA);
      }
      if (evs) cudaEventRecord(evs[1], st);
      if (kfy)
        launch_pdl(kfy, dim3((n1 + fft_yc_w(C) - 1) / fft_yc_w(C), P, B), dim3(kFftNP * fft_n1(n2)), smY, st, g, hat, yc);
      else if (y_mm)
        launch_pdl(kmy, dim3((n1 + wMy - 1) / wMy, P, B), dim3(ntMy), smMy, st, g, hat, yc, my, wMy);
      else
        launch_pdl(kb, dim3((n1 + kW - 1) / kW, P, B), dim3(yc_threads(y_fft() ? n2 : 0)), smB, st, g, hat, yc,
                   scrB);
      if (evs) cudaEventRecord(evs[2], st);
      if constexpr (std::is_same<T, float>::value)
        if (kfi) launch_pdl(kfi, dim3(n2, C, B), dim3(fft_xt_threads(n1, pmax)), smF, st, g, (const T*)hat, phi, ft);
      if (done) {
      } else if (x_mm) {
        launch_pdl(kmi, dim3(n2, C, B), dim3(ntMi), smMi, st, g, (const T*)hat, phi, mx, mti);
      } else if (split_xt) {
        launch_pdl(kct, dim3((n1 + kColsT - 1) / kColsT, n2 * C, B), dim3(kColsT), smT, st, g, hat,
                   (const T*)xt.Mt_i);
        launch_pdl(krx_i, dim3((P + kRowsX - 1) / kRowsX, n2 * C, B), dim3(256), smR, st, g, (const T*)hat, phi, xt,
                   scrS);
      } else {
        launch_pdl(kc, dim3(n2, C, B), dim3(kThreadsXt), smA, st, g, (const T*)hat, phi, xt, scrA);
      }
      if (evs) cudaEventRecord(evs[3], st);
    } else {
      if (evs) cudaEventRecord(evs[0], st);
      if (hue_mm) {
        auto xf = hue_small ? k_hue_x_fwd<T, true, kMmK> : k_hue_x_fwd<T, false, kMmK>;
        auto xi = hue_small ? k_hue_x_inv<T, true, kMmK> : k_hue_x_inv<T, false, kMmK>;
        if constexpr (sizeof(T) == 4) {
          if (hf.k == 16) xf = k_hue_x_fwd<T, false, 16>;
          if (hi.k == 16) xi = k_hue_x_inv<T, false, 16>;
        }
        launch_pdl(xf, dim3((P + hf.rb - 1) / hf.rb, hf.nch, B),
                   dim3(hf.nt), hf.smem, st, g, asrc, (const T*)f0n, (const T*)f1n, hat, mx, hf.rb, hf.chunk);
        if (evs) cudaEventRecord(evs[1], st);
        launch_pdl(hue_small ? k_hue_tt<T, true> : k_hue_tt<T, false>, dim3((n1 + hsc - 1) / hsc, B), dim3(256), smTt, st,
                   g, hat, ht, htt);
        if (evs) cudaEventRecord(evs[2], st);
        launch_pdl(xi, dim3((P + hi.rb - 1) / hi.rb, hi.nch, B),
                   dim3(hi.nt), hi.smem, st, g, (const T*)hat, phi, mx, hi.rb, hi.chunk);
      } else {
        k_hue_fwd<T><<<dim3(P, B), 256, smH, st>>>(g, asrc, f0n, f1n, hat, ht);
        if (evs) cudaEventRecord(evs[1], st);
        kh<<<dim3((n1 + 256 / pmax - 1) / (256 / pmax), B), 256, smHt, st>>>(g, hat, ht);
        if (evs) cudaEventRecord(evs[2], st);
        k_hue_inv<T><<<dim3(P, B), 256, smH, st>>>(g, hat, phi, ht);
      }
      if (evs) cudaEventRecord(evs[3], st);
    }
  }

  // partials for the largest grid the autotuner may pick (time chunks of at least 1 plane)
  size_t part_bytes() const {
    const dim3 g1 = tiled_grid(1);
    return sizeof(double) * (size_t)g1.x * g1.y * g1.z * kPart;
  }

  dim3 tiled_grid(int tchunk) const {
    // a Neumann axis leaves its last cell to the halo lane; a periodic one needs a block past it
    const int nbx = std::max(1, ((g.per1 ? n1 : n1 - 1) + kTX - 2) / (kTX - 1));
    const int nby = std::max(1, ((g.per2 ? n2 : n2 - 1) + kTY - 2) / (kTY - 1));
    const int nch = (P + tchunk - 1) / tchunk;
    return dim3(nbx, nby, B * nch);
  }

  void enqueue_update(int p, bool check, bool wx) {
    const Arrays<T> A = arrays(p, wx);
    if (tiled) {
      const dim3 grd = tiled_grid(tc);
      bool done = false;
      if constexpr (std::is_same<T, float>::value) {
        if (use_tma) {
          launch_pdl(pick_kdt(C, check, wx), grd, dim3(kTX, kTY), tma_smem(C), st, g, A, tc, part, err, tmA[p], tmB[p],
                     tmP);
          done = true;
        }
      }
      if (!done) {
        const TileLayout Lt{S, n1, n1 * n2, (long long)P * S, n1, (long long)S};
        launch_pdl(pick_kd<T>(C, check, wx, g.per1 || g.per2), grd, dim3(kTX, kTY), 0, st, g, A, tc, Lt, part);
      }
      if (check)
        k_reduce_check<<<dim3((4 + P + kReduceThreads / 32 - 1) / (kReduceThreads / 32), B), kReduceThreads, 0, st>>>(
            part, (int)(grd.x * grd.y * grd.z / B), P, acc, mass, g.active);
      return;
    }
    if (hue && !check && !wx && !g.active && B >= 8 && !plain_update) {
      // a batch of hue problems: the tiled update with the problems as its rows (no coupling between rows,
      // since the y difference factor is zero and the y components of the state stay zero); checks keep the
      // per-problem kernel below, whose sums are per problem
      Geo<T> gr = g;
      gr.n2 = B;
      gr.B = 1;
      gr.per2 = 0;
      gr.s2 = T(0);
      gr.active = nullptr;
      const TileLayout Lt{n1, P * n1, n1, 0, n1, 0};
      const int tcr = std::max(4, (P + 3) / 4);
      const dim3 grd((n1 + kTX - 2) / (kTX - 1), std::max(1, (B - 1 + kTY - 2) / (kTY - 1)), (P + tcr - 1) / tcr);
      launch_pdl(pick_kd<T>(1, false, false, true), grd, dim3(kTX, kTY), 0, st, gr, A, tcr, Lt, part);
      return;
    }
    const dim3 grd((n1 + kThreadsUpd - 1) / kThreadsUpd, n2, C * P * B);
    if (check) {
      launch_pdl(wx ? k_update<T, true, true> : k_update<T, true, false>, grd, dim3(kThreadsUpd), 0, st, g, A, acc, mass);
    } else {
      launch_pdl(wx ? k_update<T, false, true> : k_update<T, false, false>, grd, dim3(kThreadsUpd), 0, st, g, A, acc, mass);
    }
  }

  void enqueue_iteration(int p, bool check, bool wx, cudaEvent_t* evs = nullptr) {
    enqueue_poisson(p, evs);
    enqueue_update(p, check, wx);
    if (evs) cudaEventRecord(evs[4], st);
  }

  // `iters` (even) plain iterations from buffer p as one graph
  ot_status graph_for(int p, int iters = 2) {
    cudaGraphExec_t& ge = iters == 2 ? gexec[p] : glong[p];
    if (ge) return OT_OK;
    cudaGraph_t gr = nullptr;
    CUDA_OK(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    for (int i = 0; i < iters; ++i) enqueue_iteration(p ^ (i & 1), false, false);
    const cudaError_t le = cudaGetLastError();
    cudaError_t e = cudaStreamEndCapture(st, &gr);
    if (le != cudaSuccess) {
      if (gr) cudaGraphDestroy(gr);
      return seterr(OT_ECUDA, "kernel launch during graph capture: %s", cudaGetErrorString(le));
    }
    if (e != cudaSuccess) return seterr(OT_ECUDA, "graph capture: %s", cudaGetErrorString(e));
    e = cudaGraphInstantiate(&ge, gr, 0);
    cudaGraphDestroy(gr);
    if (e != cudaSuccess) return seterr(OT_ECUDA, "graph instantiate: %s", cudaGetErrorString(e));
    return OT_OK;
  }

  // plain iterations (no residual, no x output): graphs of kLongGraph iterations, then of pairs
  static constexpr int kLongGraph = 8;
  ot_status run_plain(int n) {
    while (n >= 2) {
      const int k = n >= kLongGraph ? kLongGraph : 2;
      OT_TRY(graph_for(par, k));
      CUDA_OK(cudaGraphLaunch(k == 2 ? gexec[par] : glong[par], st));
      n -= k;
    }
    if (n == 1) {
      enqueue_iteration(par, false, false);
      CUDA_OK(cudaGetLastError());
      par ^= 1;
    }
    return OT_OK;
  }

  struct Check {
    double residual = 0, energy = 0, drift = 0, dual = 0, gap = 0;
  };

  // one iteration with residuals (and x output); results land in pinned host memory
  ot_status enqueue_check(bool wx) {
    CUDA_OK(clear_results());
    enqueue_iteration(par, true, wx);
    CUDA_OK(cudaGetLastError());
    par ^= 1;
    if (wx) have_x = true;
    CUDA_OK(copy_results());
    return OT_OK;
  }

  // per-problem residual, energy (caller units) and mass drift of the last check (after a sync)
  ot_status collect_check(std::vector<ProblemCheck>& per, Check& out) {
    per.resize(B);
    out = Check{};
    if (*h_err) return seterr(OT_ETIMEOUT, "a bounded device wait of the update kernel ran out of its limit");
    for (int bi = 0; bi < B; ++bi) {
      if (g.active && !h_active[bi]) continue;   // retired: its entry keeps the check that retired it
      const double* q = &h_acc[(size_t)bi * kAcc];
      const double res = std::sqrt(q[0]) / std::max(std::sqrt(q[1]), 1e-300);
      if (!std::isfinite(res) || !std::isfinite(q[2]) || !std::isfinite(q[3]))
        return seterr(OT_ENUMERIC, "non-finite residual in problem %d", bi);
      double M = 0;
      for (int t = 0; t + 1 < P; ++t) M = std::max(M, std::fabs(h_mass[(size_t)bi * P + t] - (double)S));
      per[bi].residual = res;
      per[bi].energy = q[2] / (double)N * out_scale[bi];
      per[bi].dual = (double)g.sigma * q[3] / (double)N * out_scale[bi];
      per[bi].gap = std::fabs(per[bi].energy - per[bi].dual) /
                    std::max(std::max(std::fabs(per[bi].energy), std::fabs(per[bi].dual)), 1e-300);
      per[bi].drift = M / (double)S;
      out.residual = std::max(out.residual, res);
      out.energy += per[bi].energy / B;
      out.dual += per[bi].dual / B;
      out.gap = std::max(out.gap, per[bi].gap);
      out.drift = std::max(out.drift, per[bi].drift);
    }
    return OT_OK;
  }

  // one launch for [plain iteration on p (lead)] + check iteration (x written) + result copies
  ot_status check_graph_for(int p, bool lead) {
    if (gcheck[p][lead]) return OT_OK;
    cudaGraph_t gr = nullptr;
    CUDA_OK(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    clear_results();
    if (lead) enqueue_iteration(p, false, false);
    enqueue_iteration(lead ? 1 - p : p, true, true);
    copy_results();
    const cudaError_t le = cudaGetLastError();
    cudaError_t e = cudaStreamEndCapture(st, &gr);
    if (le != cudaSuccess) {
      if (gr) cudaGraphDestroy(gr);
      return seterr(OT_ECUDA, "launch during check-graph capture: %s", cudaGetErrorString(le));
    }
    if (e != cudaSuccess) return seterr(OT_ECUDA, "check-graph capture: %s", cudaGetErrorString(e));
    e = cudaGraphInstantiate(&gcheck[p][lead], gr, 0);
    cudaGraphDestroy(gr);
    if (e != cudaSuccess) return seterr(OT_ECUDA, "check-graph instantiate: %s", cudaGetErrorString(e));
    return OT_OK;
  }

  // n iterations, the last one a check (x written), all from graphs; results collected after a sync
  ot_status run_chunk_with_check(int n, Check& out) {
    const int plain = n - 1;
    OT_TRY(run_plain(plain - (plain & 1)));
    const bool lead = plain & 1;
    OT_TRY(check_graph_for(par, lead));
    CUDA_OK(cudaGraphLaunch(gcheck[par][lead], st));
    if (!lead) par ^= 1;   // with a lead iteration the pair returns to the same buffer
    have_x = true;
    CUDA_OK(cudaStreamSynchronize(st));
    std::vector<ProblemCheck> per;
    return collect_check(per, out);
  }

  ot_status run_check(bool wx, Check& out) {
    OT_TRY(enqueue_check(wx));
    CUDA_OK(cudaStreamSynchronize(st));
    std::vector<ProblemCheck> per;
    return collect_check(per, out);
  }

  ot_status drive(int iters, double tol, int check_every, ot_solve_stats* stats, double fallback = 0.0,
                  int* used_cold = nullptr) {
    if (iters < 1) return seterr(OT_EINVAL, "iters must be >= 1");
    CUDA_OK(cudaEventRecord(ev[10], st));
    int done = 0;
    Check ck;
    bool converged = false;
    const int K = check_every > 0 ? check_every : iters;
    while (done < iters) {
      const int chunk = std::min(K, iters - done);
      const bool last = (done + chunk == iters);
      OT_TRY(run_chunk_with_check(chunk, ck));
      const bool first = (done == 0);
      done += chunk;
      if (first && fallback > 0 && ck.residual > fallback) {
        // the warm start is worse than the threshold: restart from x = 0, b = bbar = 0
        OT_TRY(cold_start());
        if (used_cold) *used_cold = 1;
        continue;
      }
      if (tol > 0 && ck.residual <= tol) {
        converged = true;
        break;
      }
      (void)last;
    }
    CUDA_OK(cudaEventRecord(ev[11], st));
    CUDA_OK(cudaEventSynchronize(ev[11]));
    float ms = 0;
    CUDA_OK(cudaEventElapsedTime(&ms, ev[10], ev[11]));
    if (stats) {
      stats->iterations = done;
      stats->residual = ck.residual;
      stats->energy = ck.energy;
      stats->mass_drift = ck.drift;
      stats->elapsed_ms = ms;
      stats->dual_value = ck.dual;
      stats->gap = ck.gap;
    }
    if (tol > 0 && !converged) return seterr(OT_ENOTCONV, "residual %.3e > tol %.3e after %d iterations",
                                             ck.residual, tol, done);
    return OT_OK;
  }

  // ---- inputs
  ot_status load_boundary(const float* f0, const float* f1, bool normalise) {
    const size_t n = (size_t)B * S;
    CUDA_OK(cudaMemcpyAsync(stage, f0, n * sizeof(float), cudaMemcpyDefault, st));
    CUDA_OK(cudaMemcpyAsync(stage + n, f1, n * sizeof(float), cudaMemcpyDefault, st));
    return validate_scale(normalise);
  }

  // problem bi's densities into the staging area (batches assembled from separate arrays)
  ot_status stage_problem(int bi, const float* f0, const float* f1) override {
    if (bi < 0 || bi >= B || !f0 || !f1) return seterr(OT_EINVAL, "bad problem index or NULL density");
    const size_t n = (size_t)B * S;
    CUDA_OK(cudaMemcpyAsync(stage + (size_t)bi * S, f0, S * sizeof(float), cudaMemcpyDefault, st));
    CUDA_OK(cudaMemcpyAsync(stage + n + (size_t)bi * S, f1, S * sizeof(float), cudaMemcpyDefault, st));
    return OT_OK;
  }

  ot_status prepare_staged() override {
    OT_TRY(validate_scale(true));
    OT_TRY(cold_start());
    return make_dual_weights();
  }

  // validate the staged densities (section 2: f >= 0, equal masses) and rescale (reading of section 4)
  ot_status validate_scale(bool normalise) {
    const size_t n = (size_t)B * S;
    std::vector<double> sc(3 * B, 1.0);
    if (normalise) {
      CUDA_OK(cudaMemsetAsync(chk, 0, sizeof(double) * B * kChk, st));
      // minima start at +inf
      std::vector<double> init((size_t)B * kChk, 0.0);
      for (int bi = 0; bi < B; ++bi) init[(size_t)bi * kChk + 2] = init[(size_t)bi * kChk + 3] = INFINITY;
      CUDA_OK(cudaMemcpyAsync(chk, init.data(), init.size() * sizeof(double), cudaMemcpyHostToDevice, st));
      const int blocks = std::min(1024, (S + 255) / 256);
      k_check_inputs<<<dim3(blocks, B), 256, 0, st>>>(stage, stage + n, S, chk);
      CUDA_OK(cudaGetLastError());
      std::vector<double> h((size_t)B * kChk);
      CUDA_OK(cudaMemcpyAsync(h.data(), chk, h.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
      CUDA_OK(cudaStreamSynchronize(st));
      for (int bi = 0; bi < B; ++bi) {
        const double* q = &h[(size_t)bi * kChk];
        if (q[4] > 0) return seterr(OT_EMASS, "problem %d: non-finite density values", bi);
        if (q[2] < 0 || q[3] < 0) return seterr(OT_EMASS, "problem %d: negative density values", bi);
        const double M0 = q[0], M1 = q[1];
        if (!(M0 > 0) || !(M1 > 0) || std::fabs(M0 - M1) > 1e-6 * std::max(M0, M1))
          return seterr(OT_EMASS, "problem %d: masses differ (%.9g vs %.9g)", bi, M0, M1);
        sc[2 * bi] = (double)S / M0;
        sc[2 * bi + 1] = (double)S / M1;
        out_scale[bi] = 0.5 * (M0 + M1) / (double)S;
      }
    } else {
      for (int bi = 0; bi < B; ++bi) out_scale[bi] = 1.0;
    }
    for (int bi = 0; bi < B; ++bi) sc[2 * B + bi] = out_scale[bi];
    CUDA_OK(cudaMemcpyAsync(scl, sc.data(), sc.size() * sizeof(double), cudaMemcpyHostToDevice, st));
    const int blocks = std::min(1024, (S + 255) / 256);
    k_scale_boundary<T><<<dim3(blocks, B), 256, 0, st>>>(stage, stage + n, S, scl, f0n, f1n);
    CUDA_OK(cudaGetLastError());
    return OT_OK;
  }

  int grid1d(long long n) const { return (int)std::min<long long>((n + 255) / 256, 152 * 16); }

  // internal x <- packed (float), solver units
  ot_status unpack_x(const float* packed) {
    const size_t n = (size_t)B * cp.total;
    CUDA_OK(cudaMemcpyAsync(stage, packed, n * sizeof(float), cudaMemcpyDefault, st));
    k_unpack_path<T><<<grid1d((long long)B * N), 256, 0, st>>>(g, cp, stage, 1.0, x);
    CUDA_OK(cudaGetLastError());
    return OT_OK;
  }

  // w = K x0 + (0, f_b^+) for the boundary densities in f0n, f1n, with x0 = Pi_{C_d}(0) the least-norm feasible
  // path (the projection of step 1 applied to a = 0, which a[0] holds).
  ot_status make_dual_weights() {
    enqueue_poisson(0, nullptr);
    k_dual_weights<T><<<dim3(grid1d(N), B), 256, 0, st>>>(g, phi, f0n, f1n, w);
    CUDA_OK(cudaGetLastError());
    have_x = false;
    return OT_OK;
  }

  ot_status cold_start() {
    CUDA_OK(cudaMemsetAsync(a[0], 0, (size_t)B * N * sizeof(v4<T>), st));
    CUDA_OK(cudaMemsetAsync(b[0], 0, (size_t)B * N * sizeof(v4<T>), st));
    CUDA_OK(cudaMemsetAsync(b[1], 0, (size_t)B * N * sizeof(v4<T>), st));
    CUDA_OK(cudaMemsetAsync(err, 0, sizeof(int), st));
    *h_err = 0;
    par = 0;
    have_x = false;
    return OT_OK;
  }

  ot_status solve(const float* f0, const float* f1, int iters, double tol, const float* init,
                  const float* init_dual, int dual_init, double dual_support, double fallback, ot_solve_stats* stats,
                  int* used_cold) override {
    if (!f0 || !f1) return seterr(OT_EINVAL, "f0 and f1 are required");
    if (used_cold) *used_cold = 0;
    OT_TRY(load_boundary(f0, f1, true));
    OT_TRY(cold_start());
    OT_TRY(make_dual_weights());
    if (init) {
      // x0 = init (scaled to solver units per problem) into x, then b = bbar = 0 or the fixed-point dual
      const size_t n = (size_t)B * cp.total;
      CUDA_OK(cudaMemcpyAsync(stage, init, n * sizeof(float), cudaMemcpyDefault, st));
      for (int bi = 0; bi < B; ++bi) {   // one scale per problem
        Geo<T> g1 = g;
        g1.B = 1;
        const size_t off = (size_t)bi * N;
        k_unpack_path<T><<<grid1d(N), 256, 0, st>>>(g1, cp, stage + (size_t)bi * cp.total, 1.0 / out_scale[bi],
                                                    x + off);
        CUDA_OK(cudaGetLastError());
      }
      const long long cells = (long long)B * N;
      if (init_dual) {
        OT_TRY(load_dual(init_dual, b[0]));
        CUDA_OK(cudaMemcpyAsync(b[1], b[0], cells * sizeof(v4<T>), cudaMemcpyDeviceToDevice, st));
      } else if (dual_init) {
        // the domain's diameter: extent n_k / scale_k per axis, half of it on periodic axes
        double diam2 = 0;
        for (int k = 0; k < grid.ndim; ++k) {
          const double e = grid.n[k] / grid.axis_scale[k] * (grid.bc[k] == OT_BC_PERIODIC ? 0.5 : 1.0);
          diam2 += e * e;
        }
        k_dual_init<T><<<grid1d(cells), 256, 0, st>>>(g, x, f0n, f1n, T(1.0 / grid.sigma), T(1e-3),
                                                      T(std::sqrt(diam2)), T(dual_support), b[0]);
        CUDA_OK(cudaGetLastError());
        CUDA_OK(cudaMemcpyAsync(b[1], b[0], cells * sizeof(v4<T>), cudaMemcpyDeviceToDevice, st));
      }
      // a = x0 - tau sigma K^T bbar0 (bbar0 = b0)
      k_make_a<T><<<grid1d(cells), 256, 0, st>>>(g, x, b[0], a[0]);
      CUDA_OK(cudaGetLastError());
    }
    return drive(iters, tol, grid.check_every, stats, init ? fallback : 0.0, used_cold);
  }

  // ---- hooks for mixed-size batches (several plans captured into one graph)
  ot_status enqueue_pair() override {
    enqueue_iteration(par, false, false);
    enqueue_iteration(1 - par, false, false);
    CUDA_OK(cudaGetLastError());
    return OT_OK;
  }
  ot_status enqueue_single() override {
    enqueue_iteration(par, false, false);
    CUDA_OK(cudaGetLastError());
    par ^= 1;
    return OT_OK;
  }
  ot_status enqueue_check_async() override { return enqueue_check(true); }
  ot_status collect(std::vector<ProblemCheck>& per) override {
    Check ck;
    return collect_check(per, ck);
  }
  int parity() const override { return par; }

  ot_status enable_retirement() override {
    if (gexec[0] || gexec[1] || glong[0] || glong[1]) return seterr(OT_EINVAL, "retirement must be enabled before graphs are captured");
    h_active.assign(B, 1);
    CUDA_OK(cudaMemcpyAsync(active, h_active.data(), sizeof(int) * B, cudaMemcpyHostToDevice, st));
    CUDA_OK(cudaStreamSynchronize(st));
    g.active = active;
    return OT_OK;
  }
  ot_status set_active(const std::vector<int>& act, cudaStream_t s) override {
    if (!g.active || (int)act.size() != B) return seterr(OT_EINVAL, "retirement is not enabled for this plan");
    h_active = act;
    CUDA_OK(cudaMemcpyAsync(active, h_active.data(), sizeof(int) * B, cudaMemcpyHostToDevice, s));
    CUDA_OK(cudaStreamSynchronize(s));
    return OT_OK;
  }

  ot_status path_one(int bi, float* f, float* m0, float* m1, float* m2) override {
    if (!have_x) return seterr(OT_EINVAL, "no path: run a solve first");
    if (bi < 0 || bi >= B) return seterr(OT_EINVAL, "problem index out of range");
    float* ds[4] = {m0, d >= 2 ? m1 : nullptr, d >= 3 ? m2 : nullptr, f};
    Geo<T> g1 = g;
    g1.B = 1;
    const size_t off = (size_t)bi * N;
    for (int k = 0; k < 4; ++k) {
      if (!ds[k]) continue;
      float* dd[4] = {nullptr, nullptr, nullptr, nullptr};
      dd[k] = stage;
      k_pack_path<T><<<dim3(grid1d(N), 1), 256, 0, st>>>(g1, cp, x + off, scl + 2 * B + bi, nullptr, dd[0], dd[1],
                                                         dd[2], dd[3]);
      CUDA_OK(cudaGetLastError());
      CUDA_OK(cudaMemcpyAsync(ds[k], stage, (size_t)cp.len[k] * sizeof(float), cudaMemcpyDefault, st));
      CUDA_OK(cudaStreamSynchronize(st));
    }
    return OT_OK;
  }

  ot_status path(float* f, float* m0, float* m1, float* m2) override {
    if (!have_x) return seterr(OT_EINVAL, "no path: run ot_solve or ot_iterate first");
    float* ds[4] = {m0, d >= 2 ? m1 : nullptr, d >= 3 ? m2 : nullptr, f};
    for (int k = 0; k < 4; ++k) {
      if (!ds[k]) continue;
      // component k of every problem, scaled back to the caller's units
      float* dd[4] = {nullptr, nullptr, nullptr, nullptr};
      dd[k] = stage;
      k_pack_path<T><<<dim3(grid1d(N), B), 256, 0, st>>>(g, cp, x, scl + 2 * B, nullptr, dd[0], dd[1], dd[2], dd[3]);
      CUDA_OK(cudaGetLastError());
      CUDA_OK(cudaMemcpyAsync(ds[k], stage, (size_t)B * cp.len[k] * sizeof(float), cudaMemcpyDefault, st));
      CUDA_OK(cudaStreamSynchronize(st));
    }
    return OT_OK;
  }

  ot_status state_set(const float* f0, const float* f1, const float* xp, const float* bp,
                      const float* bbp) override {
    if (!f0 || !f1 || !xp || !bp) return seterr(OT_EINVAL, "f0, f1, x and b are required");
    OT_TRY(load_boundary(f0, f1, false));
    const long long cells = (long long)B * N;
    CUDA_OK(cudaMemsetAsync(a[0], 0, cells * sizeof(v4<T>), st));
    OT_TRY(make_dual_weights());
    OT_TRY(unpack_x(xp));
    CUDA_OK(cudaMemsetAsync(err, 0, sizeof(int), st));
    *h_err = 0;
    // b -> b[0]; bbar -> b[1] temporarily
    CUDA_OK(cudaMemsetAsync(b[0], 0, cells * sizeof(v4<T>), st));
    CUDA_OK(cudaMemsetAsync(b[1], 0, cells * sizeof(v4<T>), st));
    OT_TRY(load_dual(bp, b[0]));
    if (bbp) OT_TRY(load_dual(bbp, b[1]));
    else CUDA_OK(cudaMemcpyAsync(b[1], b[0], cells * sizeof(v4<T>), cudaMemcpyDeviceToDevice, st));
    // a[0] = x - tau sigma K^T bbar
    k_make_a<T><<<grid1d(cells), 256, 0, st>>>(g, x, b[1], a[0]);
    CUDA_OK(cudaGetLastError());
    // keep 2 b - bbar in b[1] so that bbar = 2 b[par] - b[1 - par] holds (all four components)
    k_axpby<T><<<grid1d(4 * cells), 256, 0, st>>>(4 * cells, T(2), (const T*)b[0], T(-1), (const T*)b[1],
                                                    (T*)b[1]);
    CUDA_OK(cudaGetLastError());
    par = 0;
    have_x = true;
    CUDA_OK(cudaStreamSynchronize(st));
    return OT_OK;
  }

  // packed dual (float, d+1 components of B*N cells... laid out problem-major) -> internal
  ot_status load_dual(const float* src, v4<T>* dst) {
    const long long cells = (long long)B * N;
    // packed dual: per problem (d+1) components of N cells
    std::vector<int> comp = comps();
    CUDA_OK(cudaMemcpyAsync(stage, src, (size_t)B * (d + 1) * N * sizeof(float), cudaMemcpyDefault, st));
    for (int bi = 0; bi < B; ++bi)
      for (int j = 0; j <= d; ++j) {
        k_comp_in<T><<<grid1d(N), 256, 0, st>>>(N, stage + ((size_t)bi * (d + 1) + j) * N, dst + (size_t)bi * N,
                                                comp[j]);
      }
    CUDA_OK(cudaGetLastError());
    (void)cells;
    return OT_OK;
  }
  std::vector<int> comps() const {
    std::vector<int> c;
    for (int k = 0; k < d; ++k) c.push_back(k);
    c.push_back(3);
    return c;
  }

  ot_status state_get(float* xp, float* bp, float* bbp) override {
    const long long cells = (long long)B * N;
    if (xp) {
      if (!have_x) return seterr(OT_EINVAL, "x is not available: run ot_iterate first");
      k_pack_path<T><<<dim3(grid1d(N), B), 256, 0, st>>>(g, cp, x, nullptr, stage, nullptr, nullptr, nullptr, nullptr);
      CUDA_OK(cudaGetLastError());
      CUDA_OK(cudaMemcpyAsync(xp, stage, (size_t)B * cp.total * sizeof(float), cudaMemcpyDefault, st));
      CUDA_OK(cudaStreamSynchronize(st));
    }
    std::vector<int> comp = comps();
    for (int which = 0; which < 2; ++which) {
      float* dst = which == 0 ? bp : bbp;
      if (!dst) continue;
      for (int bi = 0; bi < B; ++bi)
        for (int j = 0; j <= d; ++j) {
          const size_t off = (size_t)bi * N;
          float* o = stage + ((size_t)bi * (d + 1) + j) * N;
          if (which == 0) {
            k_comp_out<T><<<grid1d(N), 256, 0, st>>>(N, b[par] + off, comp[j], o);
          } else {
            // bbar = 2 b[par] - b[1-par], computed in T then converted
            k_bbar_out<T><<<grid1d(N), 256, 0, st>>>(N, b[par] + off, b[1 - par] + off, comp[j], o);
          }
        }
      CUDA_OK(cudaGetLastError());
      CUDA_OK(cudaMemcpyAsync(dst, stage, (size_t)B * (d + 1) * N * sizeof(float), cudaMemcpyDefault, st));
      CUDA_OK(cudaStreamSynchronize(st));
    }
    (void)cells;
    return OT_OK;
  }

  ot_status iterate(int iters, ot_solve_stats* stats) override { return drive(iters, 0.0, 0, stats); }

  ot_status project(const float* f0, const float* f1, const float* ap, float* xp, float* phip) override {
    if (!f0 || !f1 || !ap || !xp) return seterr(OT_EINVAL, "f0, f1, a and x are required");
    OT_TRY(load_boundary(f0, f1, false));
    OT_TRY(unpack_x(ap));
    const long long cells = (long long)B * N;
    // a[0] <- unpacked a (stored in x), run the Poisson solve, then x = a - A^T phi
    CUDA_OK(cudaMemcpyAsync(a[0], x, cells * sizeof(v4<T>), cudaMemcpyDeviceToDevice, st));
    enqueue_poisson(0, nullptr);
    Arrays<T> A = arrays(0, true);
    k_correct<T><<<grid1d(cells), 256, 0, st>>>(g, A);
    CUDA_OK(cudaGetLastError());
    k_pack_path<T><<<dim3(grid1d(N), B), 256, 0, st>>>(g, cp, x, nullptr, stage, nullptr, nullptr, nullptr, nullptr);
    CUDA_OK(cudaGetLastError());
    CUDA_OK(cudaMemcpyAsync(xp, stage, (size_t)B * cp.total * sizeof(float), cudaMemcpyDefault, st));
    if (phip) {
      k_convert<float, T><<<grid1d(cells), 256, 0, st>>>(cells, phi, stage);
      CUDA_OK(cudaMemcpyAsync(phip, stage, cells * sizeof(float), cudaMemcpyDefault, st));
    }
    CUDA_OK(cudaStreamSynchronize(st));
    have_x = false;
    return OT_OK;
  }

  ot_status profile(int iters, double ms[5]) override {
    if (iters < 1) return seterr(OT_EINVAL, "iters must be >= 1");
    double sum[4] = {0, 0, 0, 0};
    for (int i = 0; i < iters; ++i) {
      enqueue_iteration(par, false, false, ev);
      par ^= 1;
      CUDA_OK(cudaGetLastError());
      CUDA_OK(cudaEventSynchronize(ev[4]));
      for (int k = 0; k < 4; ++k) {
        float t = 0;
        CUDA_OK(cudaEventElapsedTime(&t, ev[k], ev[k + 1]));
        sum[k] += t;
      }
    }
    for (int k = 0; k < 4; ++k) ms[k] = sum[k] / iters;
    // whole iterations from the graph
    const int pairs = std::max(1, iters / 2);
    OT_TRY(graph_for(par));
    CUDA_OK(cudaGraphLaunch(gexec[par], st));  // warm
    CUDA_OK(cudaEventRecord(ev[10], st));
    for (int i = 0; i < pairs; ++i) CUDA_OK(cudaGraphLaunch(gexec[par], st));
    CUDA_OK(cudaEventRecord(ev[11], st));
    CUDA_OK(cudaEventSynchronize(ev[11]));
    float t = 0;
    CUDA_OK(cudaEventElapsedTime(&t, ev[10], ev[11]));
    ms[4] = t / (2.0 * pairs);
    return OT_OK;
  }
};


}  // namespace dynot
