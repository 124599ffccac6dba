// C ABI implementation: tape objects, device caches, launch configuration.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "compact.h"
#include "plan.h"
#include "replay.h"
#include "status.h"
#include "tape.h"

using namespace ndvm;

namespace {

thread_local std::string g_last_error;
std::mutex g_launch_mu;
unsigned long long g_launches = 0;

ndvm_status fail(ndvm_status s, const std::string& m) {
  g_last_error = m;
  return s;
}
ndvm_status cuda_fail(cudaError_t e, const char* where) {
  return fail(NDVM_E_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

struct DevPlan {
  std::vector<DevPlan> derive;  // derive plans of the shared per-point values
  DInst* code = nullptr;
  DInst* compact = nullptr;      // the compact records, or null
  DInst* matrix[2] = {nullptr, nullptr};  // the matrix records with their constants in binary64 and binary32
  DInst* code_paired = nullptr;  // the paired stream (staged and element-split variants), or null
  int32_t* args = nullptr;
  double* consts_d = nullptr;
  float* consts_f = nullptr;
};

struct DevCache {
  DevPlan grad, value;
  int* err = nullptr;
  // buffers for the host-pointer entry point: parameters, observations, losses and gradients in
  // one, and the workspace
  void* h_io = nullptr; size_t h_io_bytes = 0;
  void* h_ws = nullptr; size_t h_ws_bytes = 0;
};

}  // namespace

struct ndvm_tape {
  Tape tape;
  Plan grad_plan, value_plan;
  std::mutex mu;       // guards dev (device copies)
  std::mutex host_mu;  // serializes the host-buffer entry point and its cached buffers
  std::map<int, DevCache> dev;
};

namespace {

void free_plan(DevPlan& p) {
  for (DevPlan& d : p.derive) free_plan(d);
  cudaFree(p.code); cudaFree(p.compact); cudaFree(p.matrix[0]); cudaFree(p.matrix[1]); cudaFree(p.code_paired); cudaFree(p.args); cudaFree(p.consts_d); cudaFree(p.consts_f);
  p = DevPlan{};
}

ndvm_status upload_plan(const Tape& t, const Plan& p, DevPlan& d) {
  std::vector<double> c = t.consts;
  c.insert(c.end(), p.extra_consts.begin(), p.extra_consts.end());
  if (c.empty()) c.push_back(0.0);
  std::vector<float> cf(c.begin(), c.end());
  std::vector<int32_t> args = p.args;
  if (args.empty()) args.push_back(0);
  cudaError_t e;
  // one spare record: staged copies move 16-byte pieces and may read up to 15 bytes past the end
  if ((e = cudaMalloc(&d.code, sizeof(DInst) * (p.code.size() + 1))) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  if ((e = cudaMalloc(&d.args, sizeof(int32_t) * args.size())) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  if ((e = cudaMalloc(&d.consts_d, sizeof(double) * c.size())) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  if ((e = cudaMalloc(&d.consts_f, sizeof(float) * cf.size())) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  if (!p.code.empty() && (e = cudaMemcpy(d.code, p.code.data(), sizeof(DInst) * p.code.size(), cudaMemcpyHostToDevice)) != cudaSuccess)
    return cuda_fail(e, "cudaMemcpy");
  if (!p.code_paired.empty()) {
    if ((e = cudaMalloc(&d.code_paired, sizeof(DInst) * (p.code_paired.size() + 1))) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
    if ((e = cudaMemcpy(d.code_paired, p.code_paired.data(), sizeof(DInst) * p.code_paired.size(), cudaMemcpyHostToDevice)) != cudaSuccess)
      return cuda_fail(e, "cudaMemcpy");
  }
  if (!p.compact.empty()) {
    void* c = nullptr;
    if ((e = cudaMalloc(&c, sizeof(uint32_t) * p.compact.size())) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
    d.compact = static_cast<DInst*>(c);
    if ((e = cudaMemcpy(c, p.compact.data(), sizeof(uint32_t) * p.compact.size(), cudaMemcpyHostToDevice)) != cudaSuccess)
      return cuda_fail(e, "cudaMemcpy");
  }
  for (int f32 = 0; f32 < 2 && !p.matrix.empty(); f32++) {
    // records, constants, lists, each part padded to 16 bytes
    const size_t rb = sizeof(uint32_t) * p.matrix.size(), cb = (p.matrix_consts.size() * (f32 ? 4 : 8) + 15) / 16 * 16,
                 lb = (p.matrix_lists.size() * 4 + 15) / 16 * 16;
    std::vector<char> image(rb + cb + lb);
    std::memcpy(image.data(), p.matrix.data(), rb);
    const std::vector<float> f(p.matrix_consts.begin(), p.matrix_consts.end());
    if (f32) std::copy_n(reinterpret_cast<const char*>(f.data()), f.size() * 4, image.data() + rb);
    else std::copy_n(reinterpret_cast<const char*>(p.matrix_consts.data()), p.matrix_consts.size() * 8, image.data() + rb);
    std::copy_n(reinterpret_cast<const char*>(p.matrix_lists.data()), p.matrix_lists.size() * 4, image.data() + rb + cb);
    void* c = nullptr;
    if ((e = cudaMalloc(&c, image.size())) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
    d.matrix[f32] = static_cast<DInst*>(c);
    if ((e = cudaMemcpy(c, image.data(), image.size(), cudaMemcpyHostToDevice)) != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  }
  d.derive.resize(p.derive.size());
  for (size_t k = 0; k < p.derive.size(); k++) {
    ndvm_status s = upload_plan(t, p.derive[k], d.derive[k]);
    if (s != NDVM_OK) return s;
  }
  if ((e = cudaMemcpy(d.args, args.data(), sizeof(int32_t) * args.size(), cudaMemcpyHostToDevice)) != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  if ((e = cudaMemcpy(d.consts_d, c.data(), sizeof(double) * c.size(), cudaMemcpyHostToDevice)) != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  if ((e = cudaMemcpy(d.consts_f, cf.data(), sizeof(float) * cf.size(), cudaMemcpyHostToDevice)) != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  return NDVM_OK;
}

// device cache for the current device (uploads on first use)
ndvm_status device_cache(ndvm_tape* t, DevCache** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  std::lock_guard<std::mutex> lk(t->mu);
  auto it = t->dev.find(dev);
  if (it == t->dev.end()) {
    DevCache c;
    ndvm_status s = upload_plan(t->tape, t->grad_plan, c.grad);
    if (s == NDVM_OK) s = upload_plan(t->tape, t->value_plan, c.value);
    if (s == NDVM_OK) {
      if ((e = cudaMalloc(&c.err, sizeof(int))) != cudaSuccess) s = cuda_fail(e, "cudaMalloc");
      else if ((e = cudaMemset(c.err, 0, sizeof(int))) != cudaSuccess) s = cuda_fail(e, "cudaMemset");
    }
    if (s != NDVM_OK) {
      free_plan(c.grad); free_plan(c.value); cudaFree(c.err);
      return s;
    }
    it = t->dev.emplace(dev, c).first;
  }
  *out = &it->second;
  return NDVM_OK;
}

constexpr size_t kSmemLimit = 227 * 1024;
// per-SM resources that bound resident blocks (sm_103a): shared memory and its
// per-block reservation, registers, and the kernel's register caps (its launch
// bounds: 128 per thread for the element-split and staged variants, 64 otherwise)
constexpr size_t kSmemPerSm = 228 * 1024, kSmemPerBlockReserved = 1024;
constexpr int kRegsPerSm = 65536, kMaxRegsStagedOrShared = 128, kMaxRegsPlain = 64;
// SMs of the current device, which the launch heuristics size grids by (152 on GB300,
// also the answer when no device responds); cached per device
int64_t num_sms() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return 152;
  }
  int n = cache[dev].load(std::memory_order_relaxed);
  if (n > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    return 152;
  }
  cache[dev].store(n, std::memory_order_relaxed);
  return n;
}
// threads of a block that serves a single lane (block-cooperative matrix tapes)
constexpr int kBlockLaneThreads = 256;
// lanes per launch when a workspace is used: the kernel indexes a lane's workspace
// elements of one matrix operand with 32-bit products (element * lanes per launch)
constexpr int64_t kMaxChunk = (int64_t)1 << 22;

// Threads per lane for data-axis tapes: NDVM_THREADS_PER_LANE (1..32, a power of two)
// overrides the default, which splits a lane's points over enough threads to give
// the launch about 192 threads per SM (more threads per lane replicate the lane-level
// instructions and lengthen the reductions: 4096-lane random-expression programs on 16
// streams run 2 % faster with 8 threads per lane than with 16; 64 lanes take 32).
int threads_per_lane_override() {
  static int v = [] {
    const char* e = std::getenv("NDVM_THREADS_PER_LANE");
    int g = e ? std::atoi(e) : 0;
    return (g >= 1 && g <= 32 && (g & (g - 1)) == 0) ? g : 0;
  }();
  return v;
}

// NDVM_STAGE=0 reads the instruction stream from global memory instead of staging
// it through shared memory (a tuning knob).
bool stage_enabled() {
  static bool v = [] {
    const char* e = std::getenv("NDVM_STAGE");
    return !(e && e[0] == '0');
  }();
  return v;
}

// Launch shape of a plan: threads per block, threads per lane (1 << log2g), slot-file
// layout and shared memory per block.
struct Shape {
  int tpb = 128, log2g = 0, shared = 0, sstride = 128;
  int staged = 0, stage_off = 0;
  int points = 0;  // compact stream: points per thread and pass (0: the general kernels)
  int chunk_lanes = 0;  // lanes that a launch over part of the lanes is a multiple of
  size_t smem = 0;
};

int ilog2(int g) {
  int l = 0;
  while ((1 << l) < g) l++;
  return l;
}

// The launch shape of a compact stream; false when it does not fit.  Without a workspace, threads per
// lane and points per thread depend on the lanes and the points alone, so that a tape's value and
// gradient plans sum in the same order (tape_shape).  A gradient plan with a workspace takes the
// points one by one; its value plan, which has none, splits them, and sums in another order.
bool compact_shape(const Plan& p, size_t elem, int64_t B, Shape* out) {
  if (p.compact.empty()) return false;
  Shape s;
  const int64_t sms = num_sms();
  const size_t records = p.compact.size() / kCompactWords;
  const bool axis = p.compact_points > 0;
  // up to kCResident records are held in shared memory whole; longer streams, which have no
  // loops (compact_plan leaves those to the general kernels), are read in chunks
  const bool chunked = records > kCResident;
  s.points = 1;
  if (axis && p.n_save == 0) {
    int g = threads_per_lane_override();
    if (!g) {
      g = 1;
      while (g < 32 && B * g < sms * 192) g *= 2;
    }
    s.log2g = ilog2(g);
    if (p.compact_points > g) s.points = elem == 4 ? kPointsF32 : kPointsF64;
  }
  s.staged = chunked ? 1 : 0;
  s.sstride = p.compact_slots;
  s.stage_off = (int)(((chunked ? 2 * kCChunk : records) + 3) * kCompactWords * 4);  // (records are read ahead)
  const size_t warp_bytes = (size_t)p.compact_slots * 32 * s.points * elem;
  const int64_t warps = ((B << s.log2g) + 31) / 32;
  // threads per block: the most warps per SM at a time, then the fewest on the busiest SM
  int best_res = 0;
  int64_t best_busy = 0;
  for (int t = 128; t >= 32; t /= 2) {
    const int w = t / 32;
    const size_t smem = (size_t)s.stage_off + w * warp_bytes;
    if (smem > kSmemLimit) continue;
    const int blocks = std::min<int>((int)(kSmemPerSm / (smem + kSmemPerBlockReserved)), kRegsPerSm / (kMaxRegsStagedOrShared * t));
    const int64_t grid = (warps + w - 1) / w;
    const int64_t busy = (grid + sms - 1) / sms * w;
    const int res = (int)std::min<int64_t>((int64_t)blocks * w, busy);
    if (best_res == 0 || (busy > res ? res > best_res : best_res < best_busy ? res > best_res : busy < best_busy)) {
      best_res = res;
      best_busy = busy;
      s.tpb = t;
      s.smem = smem;
    }
  }
  if (best_res == 0) return false;
  *out = s;
  return true;
}

Shape general_shape(const Plan& p, size_t elem, int64_t B) {
  Shape s;
  const int64_t sms = num_sms();
  const int ov = threads_per_lane_override();
  if (p.has_regions && p.n_save == 0) {
    // data-axis tapes: a lane's points split over a thread group, one slot column per thread
    int g = ov;
    if (!g) {
      g = 1;
      while (g < 32 && B * g < sms * 192) g *= 2;
    }
    s.log2g = ilog2(g);
    while (s.tpb > 32 && (size_t)p.n_slots * s.tpb * elem > kSmemLimit) s.tpb /= 2;
    s.sstride = s.tpb;
  } else if (p.has_matrix) {
    // matrix tapes: G threads share a lane's slot column and split matrix elements;
    // G is large enough to give every SMSP two warps and to fit four 128-thread
    // blocks per SM in shared memory
    int g = ov > 16 ? 16 : ov;
    if (!g) {
      int gf = 1, gs = 1;
      while (gf < 16 && B * gf < sms * 4 * 64) gf *= 2;
      while (gs < 16 && (size_t)p.n_slots * (128 / gs + 1) * elem > kSmemLimit / 4) gs *= 2;
      g = gf > gs ? gf : gs;
    }
    while (g < 16 && (size_t)p.n_slots * (128 / g + 1) * elem > kSmemLimit) g *= 2;
    s.log2g = ilog2(g);
    s.shared = 1;
    // threads per block: the largest of 128, 64 and 32 whose grid spreads the lanes over
    // the SMs within 5 % of the average (the busiest SM holds ceil(blocks / SMs) blocks);
    // a 4-state filter's 8192 lanes in 16-lane blocks leave 56 SMs with 64 lanes and 96
    // with 48, in 8-lane blocks 112 SMs with 56 and 40 with 48
    auto spread = [&](int tpb) {
      const int64_t lpb = tpb >> s.log2g;
      const int64_t grid = (B + lpb - 1) / lpb;
      return (double)((grid + sms - 1) / sms * lpb) * (double)sms / (double)B;
    };
    for (int t = 128; t >= 32 && t >= g; t /= 2)
      if (spread(t) <= 1.05) { s.tpb = t; break; }
    s.sstride = (s.tpb >> s.log2g) + 1;
    if ((size_t)p.n_slots * s.sstride * elem > kSmemLimit) {
      // block-cooperative: one lane per block, whose threads split every matrix
      // instruction (large state dimensions: the lane's slot file alone fills the block)
      s.tpb = kBlockLaneThreads;
      s.log2g = ilog2(kBlockLaneThreads);
      s.sstride = 1;
    }
  } else {
    while (s.tpb > 32 && (size_t)p.n_slots * s.tpb * elem > kSmemLimit) s.tpb /= 2;
    s.sstride = s.tpb;
  }
  s.smem = (size_t)p.n_slots * s.sstride * elem;
  // long loop-free streams are staged through shared memory in double-buffered chunks,
  // unless the staging buffers would cost the launch resident blocks
  const size_t stage_bytes = 2 * kStageChunk * sizeof(DInst);
  auto blocks_per_sm = [&](size_t bytes, bool staged) {
    const int by_smem = (int)(kSmemPerSm / (bytes + kSmemPerBlockReserved));
    const int regs = (s.shared || staged) ? kMaxRegsStagedOrShared : kMaxRegsPlain;
    const int by_regs = kRegsPerSm / (regs * s.tpb);
    return by_smem < by_regs ? by_smem : by_regs;
  };
  // blocks an SM would hold at most: the grid's blocks spread over the SMs
  const int64_t lanes_per_block = s.tpb >> s.log2g;
  const int64_t grid = (B + lanes_per_block - 1) / lanes_per_block;
  const int want = (int)std::min<int64_t>((grid + sms - 1) / sms, 64);
  auto resident = [&](size_t bytes, bool staged) { return std::min(blocks_per_sm(bytes, staged), want); };
  const size_t staged_smem = (s.smem + 15) / 16 * 16 + stage_bytes;
  if (stage_enabled() && !p.has_regions && p.code.size() > 2 * (size_t)kStageChunk && staged_smem <= kSmemLimit &&
      resident(staged_smem, true) >= resident(s.smem, false)) {
    s.staged = 1;
    s.stage_off = (int)((s.smem + 15) / 16 * 16);
    s.smem = s.stage_off + stage_bytes;
  }
  return s;
}

// A replay's arguments that its plan, launch shape and type decide.
void plan_args(ReplayArgs& a, const Plan& p, const DevPlan& d, const Shape& sh, ndvm_dtype dtype, int* err) {
  // the staged and element-split variants run the paired stream; the plain one does not
  // carry the paired instruction (it would cost its register budget)
  const bool paired = (sh.staged || sh.shared) && d.code_paired != nullptr;
  const bool matrix = sh.points && sh.shared;
  a.n_consts = (int)p.matrix_consts.size();
  a.n_lists = (int)p.matrix_lists.size();
  a.code = matrix ? d.matrix[dtype == NDVM_F32] : sh.points ? d.compact : paired ? d.code_paired : d.code;
  a.n_code = (int)(matrix ? p.matrix.size() / kMatrixWords : sh.points ? p.compact.size() / kCompactWords : paired ? p.code_paired.size() : p.code.size());
  a.args = d.args;
  a.consts = dtype == NDVM_F32 ? (const void*)d.consts_f : (const void*)d.consts_d;
  a.P = p.n_params;
  a.log2g = (int16_t)sh.log2g;
  a.shared_lane = (int16_t)sh.shared;
  a.sstride = sh.sstride;
  a.staged = (int16_t)sh.staged;
  a.stage_off = sh.stage_off;
  a.points = (int16_t)sh.points;
  a.err = err;
}

// The launch shape of matrix records: the general kernels' threads per lane and per block, with
// the records' chunks, the constant matrices and the staged operands' slots in shared memory.
bool matrix_shape(const Plan& p, size_t elem, int64_t B, const Shape& g, Shape* out) {
  if (p.matrix.empty() || !g.shared) return false;
  Shape s = g;
  const size_t fixed = 2 * kMChunk * kMatrixWords * 4 + (p.matrix_consts.size() * elem + 15) / 16 * 16 +
                       (p.matrix_lists.size() * 4 + 15) / 16 * 16;
  s.points = 1;
  s.staged = 1;
  s.stage_off = (int)fixed;
  const size_t lane_bytes = (size_t)p.matrix_slots * elem;
  const bool alone = s.log2g > 5;  // the general kernel gives a lane a block: its slots fill one
  if (alone) s.log2g = 4;
  // more threads per lane where that keeps four blocks of 128 on an SM (8-state filters, 16384
  // lanes x 120 steps: 23.6 ms with 8 threads per lane, 12 warps per SM; 21.4 with 16 and 20)
  while (s.log2g < 4 && fixed + lane_bytes * (size_t)((s.tpb >> s.log2g) + 1) > kSmemLimit / 4) s.log2g++;
  // few lanes: more threads while the launch is under a warp per scheduler and each thread has
  // two elements of the largest matrix (four once a lane spans warps, whose barriers cost more)
  if (!threads_per_lane_override())
    while (s.log2g < 8 && (B << s.log2g) < num_sms() * 128 && ((s.log2g < 5 ? 4 : 8) << s.log2g) <= p.matrix_width) s.log2g++;
  // matrices of 256 elements and more: a lane alone in its block, without the padding of shared
  // rows, and threads enough for eight warps on an SM (16 states, 2000 lanes x 8 steps: 1.98 ms
  // with 16 threads per lane in 128-thread blocks, one of which fills an SM)
  if (alone || ((size_t)p.matrix_width * elem >= 2048 && !threads_per_lane_override())) s.log2g = std::max(s.log2g, 6);
  if (s.log2g > 5) {  // one lane per block
    s.smem = fixed + lane_bytes;
    if (s.smem > kSmemLimit) return false;
    const int64_t lanes = kSmemPerSm / (s.smem + kSmemPerBlockReserved);
    while (s.log2g < 8 && lanes << s.log2g < 256 && (4 << s.log2g) <= p.matrix_width) s.log2g++;
    s.tpb = 1 << s.log2g;
    s.sstride = 1;
    // the general kernel's lanes are smaller (no copies of constants): where it also has a block
    // for each and takes fewer rounds of them, it is faster (48 states in f32, 400 lanes x 4
    // steps: one round of 1.23 ms against three, 1.64 ms)
    const int64_t fit = std::min<int64_t>(kSmemPerSm / (g.smem + kSmemPerBlockReserved), kRegsPerSm / (kMaxRegsStagedOrShared * g.tpb));
    const int64_t here = std::min<int64_t>(lanes, kRegsPerSm / (kMaxRegsStagedOrShared * s.tpb)), sms = num_sms();
    if (alone && (B + fit * sms - 1) / (fit * sms) < (B + here * sms - 1) / (here * sms)) return false;
    *out = s;
    return true;
  }
  // threads per block: the general kernels', or fewer where an SM then holds more of them, or
  // more where that saves a round of blocks (9000 lanes x 10 steps of 6 states: blocks of 32 are
  // two rounds, of 128 one)
  const int64_t sms = num_sms();
  auto per_sm = [](const Shape& x) {
    return (int)std::min<int64_t>(kSmemPerSm / (x.smem + kSmemPerBlockReserved), kRegsPerSm / (kMaxRegsStagedOrShared * x.tpb));
  };
  auto rounds = [&](const Shape& x) {
    const int64_t lanes = (int64_t)per_sm(x) * (x.tpb >> x.log2g) * sms;
    return (B + lanes - 1) / lanes;
  };
  auto blocks_of = [&](int t) {
    Shape x = s;
    x.tpb = t;
    x.sstride = (t >> s.log2g) + 1;
    x.smem = fixed + lane_bytes * (size_t)x.sstride;
    return x;
  };
  const int most = std::min(std::max(g.tpb, 1 << s.log2g), 128);
  int best = 0;
  for (int t = most; t >= 32 && t >= 1 << s.log2g; t /= 2) {
    const Shape x = blocks_of(t);
    if (x.smem > kSmemLimit || per_sm(x) * t <= best) continue;
    best = per_sm(x) * t;
    s = x;
  }
  if (best == 0) return false;
  const int64_t general = rounds(g);
  for (int t = 2 * most; t <= 128 && rounds(s) > general; t *= 2) {
    const Shape x = blocks_of(t);
    if (x.smem <= kSmemLimit && rounds(x) < rounds(s)) s = x;
  }
  // The general kernel where the lanes' larger slot files (their copies of constants) add more
  // rounds than the records save: from 12 states in f64 half as many again (8000 lanes x 6 steps
  // of 12 states, five rounds against three: 2.34 ms, 2.18 by the general kernel; 4000 lanes x 10
  // steps, two against two: 1.75 and 2.58; 15 states, 9000 lanes x 6 steps, five against four:
  // 3.43 and 4.00), else twice as many of one, or of two with as many threads per lane (4000
  // lanes x 6 steps of 11 states, two against one: 1.09 ms and 0.89; 16384 lanes x 120 steps of
  // 8 states, four rounds with 16 threads per lane against two with 8: 19.3 ms and 23.6).  Behind
  // these lines: a round of records takes 0.61 to 0.69 of the general kernel's with as many threads
  // per lane (the pairs above) and 0.41 with twice as many; they move when a kernel does.
  if (elem == 8 && p.matrix_width >= 128 && 2 * rounds(s) >= 3 * general) return false;
  if (s.log2g >= 3 && rounds(s) >= 2 * general && (general == 1 || (general == 2 && s.log2g == g.log2g))) return false;
  *out = s;
  return true;
}

// A partial launch (a workspace smaller than all lanes need) covers a multiple of the general
// kernels' lanes per block, whichever kernel runs: the smallest workspace a call accepts
// depends on the tape and its lanes only.
Shape launch_shape(const Plan& p, size_t elem, int64_t B) {
  const Shape g = general_shape(p, elem, B);
  Shape s = g;
  if (!matrix_shape(p, elem, B, g, &s) && !compact_shape(p, elem, B, &s)) s = g;
  s.chunk_lanes = g.tpb >> g.log2g;
  return s;
}

// The same of a tape's gradient or value plan.  A data sum's points are added in the order of the
// kernel that runs them, so the value plan runs on the general one where the gradient plan's slots do
// not fit the other.
Shape tape_shape(const ndvm_tape* t, bool grad, size_t elem, int64_t B) {
  const Plan &g = t->grad_plan, &v = t->value_plan;
  Shape s = launch_shape(grad ? g : v, elem, B);
  if (!grad && s.points && v.compact_points > 0 && g.n_save == 0 && !launch_shape(g, elem, B).points) {
    const int chunk_lanes = s.chunk_lanes;
    s = general_shape(v, elem, B);
    s.chunk_lanes = chunk_lanes;
  }
  return s;
}

// bytes of the extended observations (a copy of the observations the program reads,
// then the regions' blocks of shared per-point values), rounded up to 256; 0 without
size_t derived_bytes(const Plan& p, size_t elem) {
  if (p.derive.empty()) return 0;
  return ((size_t)(p.n_obs_min + p.derived_elems) * elem + 255) / 256 * 256;
}

// Compact streams read the observations where they are, and the regions' blocks from the extended
// ones (args, which scalar records do not use, points to them); the general kernels find both there.
bool reads_both(const Shape& sh) { return sh.points > 0 && !sh.shared; }

void set_obs(ReplayArgs& a, const Shape& sh, const void* obs, const void* ext) {
  if (ext && reads_both(sh)) a.args = static_cast<const int32_t*>(ext);
  a.obs = ext && !reads_both(sh) ? ext : obs;
}

// Fill the extended observations at `ext`: copy obs[0 .. n_obs_min) if `copy`, then run the derive
// plans, one lane per point of each region, each lane's parameters being its point's
// observation record (params = obs + base, P = stride).
ndvm_status run_derive(const Plan& p, const DevPlan& dp, ndvm_dtype dtype, const void* obs, void* ext, bool copy,
                       int* err, void* stream) {
  const size_t elem = dtype == NDVM_F32 ? sizeof(float) : sizeof(double);
  cudaError_t e = cudaSuccess;
  if (copy) e = cudaMemcpyAsync(ext, obs, (size_t)p.n_obs_min * elem, cudaMemcpyDeviceToDevice, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "copy observations");
  for (size_t k = 0; k < p.derive.size(); k++) {
    const Plan& q = p.derive[k];
    const DeriveInfo& di = p.derive_info[k];
    const DevPlan& dq = dp.derive[k];
    if (di.n_points <= 0) continue;
    const Shape sh = launch_shape(q, elem, di.n_points);
    ReplayArgs a;
    plan_args(a, q, dq, sh, dtype, err);
    a.obs = obs;
    a.params = static_cast<const char*>(obs) + (size_t)di.base * elem;
    a.loss = nullptr;
    a.grad = nullptr;
    a.save = static_cast<char*>(ext) + (size_t)(p.n_obs_min + di.offset) * elem;
    a.save_ld = di.n_points;
    a.P = (int)di.stride;
    a.lane0 = 0;
    a.lane_end = di.n_points;
    const int64_t lanes_per_block = sh.tpb >> sh.log2g;
    const int64_t blocks = (di.n_points + lanes_per_block - 1) / lanes_per_block;
    {
      std::lock_guard<std::mutex> lk(g_launch_mu);
      e = launch_replay(a, dtype == NDVM_F32, (int)blocks, sh.tpb, sh.smem, (cudaStream_t)stream);
      g_launches++;
    }
    if (e != cudaSuccess) return cuda_fail(e, "derive launch");
  }
  return NDVM_OK;
}

ndvm_status run(ndvm_tape* t, bool grad, ndvm_dtype dtype, int64_t B, const void* params, const void* obs,
                int64_t n_obs, void* loss, void* gradp, void* ws, size_t ws_bytes, void* stream) {
  if (!t) return fail(NDVM_E_INVALID_ARG, "null tape");
  if (dtype != NDVM_F64 && dtype != NDVM_F32) return fail(NDVM_E_INVALID_ARG, "bad dtype");
  if (B < 0) return fail(NDVM_E_INVALID_ARG, "B must be >= 0");
  if (B == 0) return NDVM_OK;
  const Plan& p = grad ? t->grad_plan : t->value_plan;
  if (B > (int64_t)1 << 40) return fail(NDVM_E_INVALID_ARG, "B too large");
  if (p.n_params > 0 && !params) return fail(NDVM_E_INVALID_ARG, "null params");
  if (!loss) return fail(NDVM_E_INVALID_ARG, "null loss");
  if (grad && p.n_params > 0 && !gradp) return fail(NDVM_E_INVALID_ARG, "null grad");
  if (n_obs < p.n_obs_min) return fail(NDVM_E_INVALID_ARG, "obs holds " + std::to_string(n_obs) + " values but the program reads " + std::to_string(p.n_obs_min));
  if (p.n_obs_min > 0 && !obs) return fail(NDVM_E_INVALID_ARG, "null obs");
  const size_t elem = dtype == NDVM_F32 ? sizeof(float) : sizeof(double);
  const Shape sh = tape_shape(t, grad, elem, B);
  const int tpb = sh.tpb, log2g = sh.log2g;
  const size_t smem = sh.smem;
  if (smem > kSmemLimit) return fail(NDVM_E_UNSUPPORTED, "tape needs " + std::to_string(p.n_slots) + " slots per lane, more than shared memory holds");
  const int lanes_per_block = tpb >> log2g;
  // the workspace holds the shared per-point values first, then the per-lane saves
  const size_t der_bytes = grad ? derived_bytes(p, elem) : 0;
  if (der_bytes > 0 && (!ws || ws_bytes < der_bytes))
    return fail(NDVM_E_INVALID_ARG, "this tape needs a workspace of at least " + std::to_string(der_bytes) + " bytes");
  void* lane_ws = der_bytes > 0 ? static_cast<char*>(ws) + der_bytes : ws;
  if (der_bytes > 0) ws_bytes -= der_bytes;
  int64_t chunk = B;
  if (grad && p.n_save > 0) {
    const size_t per_lane = (size_t)p.n_save * elem;
    if (!ws) return fail(NDVM_E_INVALID_ARG, "this tape needs a workspace of " + std::to_string(per_lane) + " bytes per lane");
    int64_t fit = (int64_t)(ws_bytes / per_lane);
    if (fit > kMaxChunk) fit = kMaxChunk;
    if (fit < B) {
      fit -= fit % sh.chunk_lanes;
      if (fit < sh.chunk_lanes)
        return fail(NDVM_E_INVALID_ARG, "workspace too small: need at least " + std::to_string(per_lane * sh.chunk_lanes) + " bytes");
      chunk = fit;
    }
  }
  DevCache* dc = nullptr;
  ndvm_status s = device_cache(t, &dc);
  if (s != NDVM_OK) return s;
  const DevPlan& dp = grad ? dc->grad : dc->value;
  if (der_bytes > 0 && (s = run_derive(p, dp, dtype, obs, ws, !reads_both(sh), dc->err, stream)) != NDVM_OK) return s;
  ReplayArgs a;
  plan_args(a, p, dp, sh, dtype, dc->err);
  set_obs(a, sh, obs, der_bytes > 0 ? ws : nullptr);
  a.params = params;
  a.loss = loss;
  a.grad = gradp;
  a.save = lane_ws;
  a.save_ld = chunk;
  for (int64_t l0 = 0; l0 < B; l0 += chunk) {
    a.lane0 = l0;
    a.lane_end = l0 + chunk < B ? l0 + chunk : B;
    const int64_t lanes = a.lane_end - l0;
    const int64_t blocks = (lanes + lanes_per_block - 1) / lanes_per_block;
    if (blocks > 0x7fffffff) return fail(NDVM_E_INVALID_ARG, "too many lanes for one launch");
    cudaError_t e;
    {
      std::lock_guard<std::mutex> lk(g_launch_mu);
      e = launch_replay(a, dtype == NDVM_F32, (int)blocks, tpb, smem, (cudaStream_t)stream);
      g_launches++;
    }
    if (e != cudaSuccess) return cuda_fail(e, "replay launch");
  }
  return NDVM_OK;
}

// resident blocks per SM of a launch shape (shared memory and registers)
int resident_blocks(const Shape& s) {
  const int by_smem = (int)(kSmemPerSm / (s.smem + kSmemPerBlockReserved));
  const int regs = (s.shared || s.staged || s.points) ? kMaxRegsStagedOrShared : kMaxRegsPlain;
  const int by_regs = kRegsPerSm / (regs * s.tpb);
  return std::max(1, std::min(by_smem, by_regs));
}

// One replay of a batched launch: its arguments, its blocks and its launch shape.
struct Member {
  ReplayArgs a;
  int64_t blocks;
  Shape sh;
  std::array<int, 6> key;  // what members of one launch have in common (last: resident blocks per SM)

  explicit Member(const Shape& s) : sh(s), key{s.shared, s.staged, s.log2g, s.tpb, s.points, resident_blocks(s)} {}
};

// Launches the members in as few kernels as possible: one per run of members with the
// same kernel variant, block size and threads per lane.  The launch's shared memory is its largest
// member's, which may cost the others resident blocks: members of different resident blocks per
// SM share a launch while it has at most kMergeRounds times the blocks that are on the SMs at once.
// Launches follow each other on the stream, and each ends with its slowest blocks on a nearly idle
// chip; blocks of one launch follow each other without that, the longest programs' first.
// Random expressions, us per call with one round, two, four, sixteen: 24 programs x 300 lanes x 256
// points 298, 274, 261, 263; 8 x 1000 x 256 290, 257, 248, 228; 16 x 2000 x 128 570, 510, 467, 441;
// 30 x 700 x 200 700, 613, 614, 703; 24 x 4096 x 256 2690, 2537, 2503, 2655.  At most kMultiMax
// members and 2^31 - 1 blocks per launch.
constexpr int64_t kMergeRounds = 4;
ndvm_status launch_members(std::vector<Member>& ms, bool f32, void* stream) {
  std::stable_sort(ms.begin(), ms.end(), [](const Member& x, const Member& y) { return x.key < y.key; });
  // (within a kind, fewest resident blocks -- most shared memory -- first)
  for (size_t i = 0; i < ms.size();) {
    const std::array<int, 6> k = ms[i].key;
    int64_t blocks = 0;
    size_t j = i;
    for (; j < ms.size() && std::equal(k.begin(), k.end() - 1, ms[j].key.begin()); j++) {
      if (ms[j].key != k && blocks + ms[j].blocks > kMergeRounds * num_sms() * k.back()) break;
      blocks += ms[j].blocks;
    }
    for (size_t q = i; q < j; q++) ms[q].key = k;
    // (the longest programs' blocks start first)
    std::stable_sort(ms.begin() + (int64_t)i, ms.begin() + (int64_t)j,
                     [](const Member& x, const Member& y) { return x.a.n_code > y.a.n_code; });
    i = j;
  }
  std::unique_ptr<MultiArgs> table(new MultiArgs);  // about 31 KB: on the heap
  for (size_t i = 0; i < ms.size();) {
    MultiArgs& m = *table;
    m.n = 0;
    int64_t blocks = 0;
    size_t smem = 0;
    const std::array<int, 6> k = ms[i].key;
    while (i < ms.size() && m.n < kMultiMax && ms[i].key == k && blocks + ms[i].blocks <= 0x7fffffff) {
      m.start[m.n] = (int)blocks;
      m.a[m.n] = ms[i].a;
      blocks += ms[i].blocks;
      smem = std::max(smem, ms[i].sh.smem);
      m.n++;
      i++;
    }
    if (m.n == 0) return fail(NDVM_E_INVALID_ARG, "too many lanes for one launch");
    m.start[m.n] = (int)blocks;
    cudaError_t e;
    {
      std::lock_guard<std::mutex> lk(g_launch_mu);
      e = launch_replay_multi(m, f32, (int)blocks, k[3], smem, (cudaStream_t)stream);
      g_launches++;
    }
    if (e != cudaSuccess) return cuda_fail(e, "batched replay launch");
  }
  return NDVM_OK;
}

// Workspace of a batch: per tape with lanes, a 256-byte aligned region holding its
// extended observations (shared per-point values) and then its lanes' saved values.
// Returns the bytes needed; offsets[k] receives tape k's region (relative to the base).
size_t multi_layout(ndvm_tape* const* tapes, int32_t n, const int64_t* B, size_t elem, std::vector<size_t>* offsets) {
  size_t cur = 0;
  for (int32_t k = 0; k < n; k++) {
    size_t off = 0;
    if (tapes[k] && B[k] > 0) {
      const Plan& p = tapes[k]->grad_plan;
      const size_t need = derived_bytes(p, elem) + (size_t)p.n_save * elem * (size_t)B[k];
      if (need > 0) {
        cur = (cur + 255) / 256 * 256;
        off = cur;
        cur += need;
      }
    }
    if (offsets) offsets->push_back(off);
  }
  return cur;
}

ndvm_status run_multi(ndvm_tape* const* tapes, int32_t n, ndvm_dtype dtype, const int64_t* B,
                      const void* const* params, const void* const* obs, const int64_t* n_obs, void* const* loss,
                      void* const* grad, void* ws, size_t ws_bytes, void* stream) {
  if (n < 0) return fail(NDVM_E_INVALID_ARG, "negative tape count");
  if (n == 0) return NDVM_OK;
  if (!tapes || !B || !params || !obs || !n_obs || !loss || !grad) return fail(NDVM_E_INVALID_ARG, "null argument array");
  if (dtype != NDVM_F64 && dtype != NDVM_F32) return fail(NDVM_E_INVALID_ARG, "bad dtype");
  if (ws && (reinterpret_cast<uintptr_t>(ws) & 255)) return fail(NDVM_E_INVALID_ARG, "workspace must be 256-byte aligned");
  const size_t elem = dtype == NDVM_F32 ? sizeof(float) : sizeof(double);
  std::vector<Shape> shapes((size_t)n);
  for (int32_t k = 0; k < n; k++) {
    auto refuse = [k](ndvm_status s, const char* m) { return fail(s, std::string(m) + " (tape " + std::to_string(k) + ")"); };
    if (!tapes[k]) return refuse(NDVM_E_INVALID_ARG, "null tape");
    if (B[k] < 0) return refuse(NDVM_E_INVALID_ARG, "B must be >= 0");
    if (B[k] > (int64_t)1 << 40) return refuse(NDVM_E_INVALID_ARG, "B too large");
    if (B[k] == 0) continue;
    const Plan& p = tapes[k]->grad_plan;
    if (p.n_params > 0 && (!params[k] || !grad[k])) return refuse(NDVM_E_INVALID_ARG, "null params or grad");
    if (!loss[k]) return refuse(NDVM_E_INVALID_ARG, "null loss");
    if (n_obs[k] < p.n_obs_min) return refuse(NDVM_E_INVALID_ARG, "obs holds too few values");
    if (p.n_obs_min > 0 && !obs[k]) return refuse(NDVM_E_INVALID_ARG, "null obs");
    shapes[(size_t)k] = launch_shape(p, elem, B[k]);
    if (shapes[(size_t)k].smem > kSmemLimit)
      return refuse(NDVM_E_UNSUPPORTED, "tape needs more slots per lane than shared memory holds");
  }
  std::vector<size_t> off;
  const size_t need = multi_layout(tapes, n, B, elem, &off);
  if (need > 0 && (!ws || ws_bytes < need))
    return fail(NDVM_E_INVALID_ARG, "this batch needs a workspace of " + std::to_string(need) + " bytes");
  std::vector<Member> main, der;
  std::unique_ptr<CopyRuns> runs(new CopyRuns);
  runs->n = 0;
  std::vector<CopyRuns> run_batches;
  for (int32_t k = 0; k < n; k++) {
    if (B[k] == 0) continue;
    ndvm_tape* t = tapes[k];
    const Plan& p = t->grad_plan;
    DevCache* dc = nullptr;
    ndvm_status st = device_cache(t, &dc);
    if (st != NDVM_OK) return st;
    const DevPlan& dp = dc->grad;
    char* base = static_cast<char*>(ws) + off[(size_t)k];
    const size_t der_bytes = derived_bytes(p, elem);
    if (der_bytes > 0) {
      // the observations the program reads, then the derive plans (one lane per point)
      if (p.n_obs_min > 0 && !reads_both(shapes[(size_t)k])) {
        if (runs->n == kCopyRunsMax) { run_batches.push_back(*runs); runs->n = 0; }
        runs->src[runs->n] = obs[k];
        runs->dst[runs->n] = base;
        runs->words[runs->n] = (int64_t)((size_t)p.n_obs_min * elem / 4);
        runs->n++;
      }
      for (size_t q = 0; q < p.derive.size(); q++) {
        const Plan& dq = p.derive[q];
        const DeriveInfo& di = p.derive_info[q];
        const DevPlan& dd = dp.derive[q];
        if (di.n_points <= 0) continue;
        Member m(launch_shape(dq, elem, di.n_points));
        ReplayArgs& a = m.a;
        plan_args(a, dq, dd, m.sh, dtype, dc->err);
        a.obs = obs[k];
        a.params = static_cast<const char*>(obs[k]) + (size_t)di.base * elem;
        a.loss = nullptr;
        a.grad = nullptr;
        a.save = base + (size_t)(p.n_obs_min + di.offset) * elem;
        a.save_ld = di.n_points;
        a.P = (int)di.stride;
        a.lane0 = 0;
        a.lane_end = di.n_points;
        const int64_t lpb = m.sh.tpb >> m.sh.log2g;
        m.blocks = (di.n_points + lpb - 1) / lpb;
        der.push_back(m);
      }
    }
    // (members of at most kMaxChunk lanes where they use the workspace, each a part of its own)
    const int64_t chunk = p.n_save > 0 ? std::min(B[k], kMaxChunk) : B[k];
    for (int64_t l0 = 0; l0 < B[k]; l0 += chunk) {
      Member m(shapes[(size_t)k]);
      ReplayArgs& a = m.a;
      plan_args(a, p, dp, m.sh, dtype, dc->err);
      set_obs(a, m.sh, obs[k], der_bytes > 0 ? base : nullptr);
      a.params = params[k];
      a.loss = loss[k];
      a.grad = grad[k];
      a.lane0 = l0;
      a.lane_end = std::min(l0 + chunk, B[k]);
      const int64_t lanes = a.lane_end - l0, lpb = m.sh.tpb >> m.sh.log2g;
      a.save = base + der_bytes + (size_t)l0 * (size_t)p.n_save * elem;
      a.save_ld = lanes;
      m.blocks = (lanes + lpb - 1) / lpb;
      if (m.blocks > 0x7fffffff) return fail(NDVM_E_INVALID_ARG, "too many lanes for one launch");
      main.push_back(m);
    }
  }
  if (runs->n > 0) run_batches.push_back(*runs);
  for (const CopyRuns& c : run_batches) {
    cudaError_t e;
    {
      std::lock_guard<std::mutex> lk(g_launch_mu);
      e = launch_copy_runs(c, (cudaStream_t)stream);
      g_launches++;
    }
    if (e != cudaSuccess) return cuda_fail(e, "observation copies");
  }
  ndvm_status st = launch_members(der, dtype == NDVM_F32, stream);
  if (st != NDVM_OK) return st;
  return launch_members(main, dtype == NDVM_F32, stream);
}

ndvm_status ensure(void** buf, size_t* have, size_t need) {
  if (*have >= need && *buf) return NDVM_OK;
  cudaFree(*buf);
  *buf = nullptr;
  *have = 0;
  cudaError_t e = cudaMalloc(buf, need ? need : 16);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? fail(NDVM_E_OOM, "device allocation failed") : cuda_fail(e, "cudaMalloc");
  *have = need;
  return NDVM_OK;
}

}  // namespace

extern "C" {

ndvm_status ndvm_trace_build(const char* program, size_t len, ndvm_frontend fe, ndvm_tape** out) {
  if (!program || !out) return fail(NDVM_E_INVALID_ARG, "null argument");
  if (fe != NDVM_FE_SCHEME && fe != NDVM_FE_BYTECODE) return fail(NDVM_E_INVALID_ARG, "unknown front end");
  *out = nullptr;
  try {
    Builder b;
    std::string err;
    if (fe == NDVM_FE_SCHEME) trace_scheme(program, len, b, err);
    else trace_bytecode(program, len, b, err);
    if (b.t.loss < 0) return fail(NDVM_E_PARSE, "program produced no result");
    ndvm_tape* t = new ndvm_tape();
    t->tape = std::move(b.t);
    t->grad_plan = make_plan(t->tape, true);
    t->value_plan = make_plan(t->tape, false);
    std::string why;
    if (!validate_plan(t->grad_plan, t->tape.consts.size(), why) || !validate_plan(t->value_plan, t->tape.consts.size(), why)) {
      delete t;
      return fail(NDVM_E_UNSUPPORTED, "internal plan check failed: " + why);
    }
    // (of checked plans: the translation indexes their lists and constants)
    compact_plan(t->grad_plan, t->tape.consts);
    compact_plan(t->value_plan, t->tape.consts);
    // (both or neither, where both split a data sum's points: its order of addition is the kernel's)
    Plan &g = t->grad_plan, &v = t->value_plan;
    if (g.has_regions && g.n_save == 0 && g.compact.empty() != v.compact.empty()) {
      g.compact.clear();
      v.compact.clear();
    }
    *out = t;
    return NDVM_OK;
  } catch (const BuildError& e) {
    return fail((ndvm_status)e.code, e.msg);
  } catch (const std::bad_alloc&) {
    return fail(NDVM_E_OOM, "host allocation failed");
  } catch (const std::exception& e) {
    return fail(NDVM_E_UNSUPPORTED, e.what());
  }
}

ndvm_status ndvm_tape_info(const ndvm_tape* t, int64_t* n_nodes, int32_t* n_params, int64_t* n_obs, int64_t* n_slots,
                           uint64_t* hash) {
  if (!t) return fail(NDVM_E_INVALID_ARG, "null tape");
  if (n_nodes) *n_nodes = (int64_t)t->tape.nodes.size();
  if (n_params) *n_params = t->tape.n_params;
  if (n_obs) *n_obs = t->tape.n_obs_min;
  if (n_slots) *n_slots = t->grad_plan.n_slots;
  if (hash) *hash = t->tape.hash();
  return NDVM_OK;
}

ndvm_status ndvm_tape_cost(const ndvm_tape* t, double* work_fwd, double* work_rev, int64_t* save_elems,
                           int32_t* flags) {
  if (!t) return fail(NDVM_E_INVALID_ARG, "null tape");
  const Plan& p = t->grad_plan;
  const bool records = !p.compact.empty() || !p.matrix.empty();
  if (work_fwd) *work_fwd = p.work_fwd + (records ? p.records_fwd : 0);
  if (work_rev) *work_rev = p.work_rev + (records ? p.records_rev : 0);
  if (save_elems) *save_elems = p.n_save;
  if (flags) *flags = (p.has_regions ? 1 : 0) | (p.spill ? 2 : 0);
  return NDVM_OK;
}

ndvm_status ndvm_tape_shared_work(const ndvm_tape* t, double* work_per_call) {
  if (!t || !work_per_call) return fail(NDVM_E_INVALID_ARG, "null argument");
  double w = 0;
  for (const DeriveInfo& di : t->grad_plan.derive_info) w += di.work * (double)di.n_points;
  *work_per_call = w;
  return NDVM_OK;
}

ndvm_status ndvm_tape_serialize(const ndvm_tape* t, void* buf, size_t cap, size_t* len) {
  if (!t || !len) return fail(NDVM_E_INVALID_ARG, "null argument");
  std::vector<uint8_t> s = t->tape.serialize();
  *len = s.size();
  if (!buf && cap == 0) return NDVM_OK;
  if (!buf || cap < s.size()) return fail(NDVM_E_INVALID_ARG, "buffer too small");
  std::memcpy(buf, s.data(), s.size());
  return NDVM_OK;
}

void ndvm_tape_free(ndvm_tape* t) {
  if (!t) return;
  int cur = 0;
  cudaGetDevice(&cur);
  for (auto& kv : t->dev) {
    cudaSetDevice(kv.first);
    DevCache& c = kv.second;
    free_plan(c.grad); free_plan(c.value);
    cudaFree(c.err);
    cudaFree(c.h_io); cudaFree(c.h_ws);
  }
  if (!t->dev.empty()) cudaSetDevice(cur);
  delete t;
}

size_t ndvm_workspace_bytes(const ndvm_tape* t, int64_t B, ndvm_dtype dtype) {
  if (!t || B <= 0) return 0;
  size_t elem = dtype == NDVM_F32 ? sizeof(float) : sizeof(double);
  return derived_bytes(t->grad_plan, elem) + (size_t)t->grad_plan.n_save * elem * (size_t)B;
}

ndvm_status ndvm_forward(const ndvm_tape* tape, ndvm_dtype dtype, int64_t B, const void* params, const void* obs,
                         int64_t n_obs, void* loss, void* stream) {
  return run(const_cast<ndvm_tape*>(tape), false, dtype, B, params, obs, n_obs, loss, nullptr, nullptr, 0, stream);
}

ndvm_status ndvm_value_and_grad(const ndvm_tape* tape, ndvm_dtype dtype, int64_t B, const void* params,
                                const void* obs, int64_t n_obs, void* loss, void* grad, void* ws, size_t ws_bytes,
                                void* stream) {
  return run(const_cast<ndvm_tape*>(tape), true, dtype, B, params, obs, n_obs, loss, grad, ws, ws_bytes, stream);
}

size_t ndvm_workspace_bytes_multi(const ndvm_tape* const* tapes, int32_t n_tapes, const int64_t* B, ndvm_dtype dtype) {
  if (!tapes || !B || n_tapes <= 0) return 0;
  for (int32_t k = 0; k < n_tapes; k++)
    if (B[k] < 0) return 0;
  return multi_layout(const_cast<ndvm_tape* const*>(tapes), n_tapes, B, dtype == NDVM_F32 ? sizeof(float) : sizeof(double),
                      nullptr);
}

ndvm_status ndvm_value_and_grad_multi(const ndvm_tape* const* tapes, int32_t n_tapes, ndvm_dtype dtype, const int64_t* B,
                                      const void* const* params, const void* const* obs, const int64_t* n_obs,
                                      void* const* loss, void* const* grad, void* workspace, size_t ws_bytes,
                                      void* stream) {
  try {
    return run_multi(const_cast<ndvm_tape* const*>(tapes), n_tapes, dtype, B, params, obs, n_obs, loss, grad, workspace,
                     ws_bytes, stream);
  } catch (const std::bad_alloc&) {
    return fail(NDVM_E_OOM, "host allocation failed");
  }
}

}  // extern "C"

namespace {

// host-buffer replay: copies in, replay, copies out, on one stream; `sync` waits for them
// Host memory that CUDA does not know.
bool is_pageable(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) == cudaSuccess) return a.type == cudaMemoryTypeUnregistered;
  cudaGetLastError();
  return false;
}

ndvm_status host_replay(const ndvm_tape* tape, ndvm_dtype dtype, int64_t B, const void* params, const void* obs,
                        int64_t n_obs, void* loss, void* grad, void* stream, bool sync) {
  ndvm_tape* t = const_cast<ndvm_tape*>(tape);
  if (!t) return fail(NDVM_E_INVALID_ARG, "null tape");
  if (B < 0 || n_obs < 0) return fail(NDVM_E_INVALID_ARG, "negative size");
  if (B == 0) return NDVM_OK;
  if (!loss || (t->tape.n_params > 0 && !params) || (n_obs > 0 && !obs)) return fail(NDVM_E_INVALID_ARG, "null argument");
  DevCache* dc = nullptr;
  ndvm_status s = device_cache(t, &dc);
  if (s != NDVM_OK) return s;
  const size_t elem = dtype == NDVM_F32 ? sizeof(float) : sizeof(double);
  const size_t pb = (size_t)B * t->tape.n_params * elem, ob = (size_t)n_obs * elem, lb = (size_t)B * elem;
  const bool want_grad = grad != nullptr;
  size_t wsb = want_grad ? ndvm_workspace_bytes(t, B, dtype) : 0;
  std::lock_guard<std::mutex> lk(t->host_mu);
  const size_t gb = want_grad ? pb : 0;
  auto pad = [](size_t n) { return (n + 255) / 256 * 256; };
  const size_t in = pad(pb) + ob, out = pad(lb) + gb;  // two runs: inputs, then outputs
  if ((s = ensure(&dc->h_io, &dc->h_io_bytes, pad(in) + out)) != NDVM_OK) return s;
  if (wsb && (s = ensure(&dc->h_ws, &dc->h_ws_bytes, wsb)) != NDVM_OK) return s;
  char* d_params = static_cast<char*>(dc->h_io);
  char* d_obs = d_params + pad(pb);
  char* d_loss = d_params + pad(in);
  char* d_grad = d_loss + pad(lb);
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e;
  // A synchronous call's small inputs and outputs travel as one copy each way, through a buffer of
  // this call: a transfer's fixed cost (about 8 us) is more than copying 64 KB on the host.  Not so
  // inputs in page-locked or managed memory: earlier work on the stream may still write them, and
  // copies on the stream come after it.
  constexpr size_t kOneCopy = 64 * 1024;
  std::vector<char> host;
  if (sync && pb && ob && in <= kOneCopy && is_pageable(params) && is_pageable(obs)) {
    host.resize(in);
    std::memcpy(host.data(), params, pb);
    std::memcpy(host.data() + pad(pb), obs, ob);
    if ((e = cudaMemcpyAsync(d_params, host.data(), in, cudaMemcpyHostToDevice, st)) != cudaSuccess) return cuda_fail(e, "copy inputs");
  } else {
    if (pb && (e = cudaMemcpyAsync(d_params, params, pb, cudaMemcpyHostToDevice, st)) != cudaSuccess) return cuda_fail(e, "copy params");
    if (ob && (e = cudaMemcpyAsync(d_obs, obs, ob, cudaMemcpyHostToDevice, st)) != cudaSuccess) return cuda_fail(e, "copy obs");
  }
  if (want_grad)
    s = run(t, true, dtype, B, d_params, n_obs ? d_obs : nullptr, n_obs, d_loss, d_grad, dc->h_ws, wsb, stream);
  else
    s = run(t, false, dtype, B, d_params, n_obs ? d_obs : nullptr, n_obs, d_loss, nullptr, nullptr, 0, stream);
  if (s != NDVM_OK) {
    if (!host.empty()) cudaStreamSynchronize(st);  // (the copy may still read this call's buffer)
    return s;
  }
  if (sync && gb && out <= kOneCopy) {
    std::vector<char> back(out);
    if ((e = cudaMemcpyAsync(back.data(), d_loss, out, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return cuda_fail(e, "copy outputs");
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_fail(e, "synchronize");
    std::memcpy(loss, back.data(), lb);
    std::memcpy(grad, back.data() + pad(lb), gb);
    return NDVM_OK;
  }
  if ((e = cudaMemcpyAsync(loss, d_loss, lb, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return cuda_fail(e, "copy loss");
  if (gb && (e = cudaMemcpyAsync(grad, d_grad, gb, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return cuda_fail(e, "copy grad");
  if (sync && (e = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_fail(e, "synchronize");
  return NDVM_OK;
}

}  // namespace

extern "C" {

ndvm_status ndvm_value_and_grad_host(const ndvm_tape* tape, ndvm_dtype dtype, int64_t B, const void* params,
                                     const void* obs, int64_t n_obs, void* loss, void* grad, void* stream) {
  try {
    return host_replay(tape, dtype, B, params, obs, n_obs, loss, grad, stream, true);
  } catch (const std::bad_alloc&) {
    return fail(NDVM_E_OOM, "host allocation failed");
  }
}

ndvm_status ndvm_value_and_grad_host_async(const ndvm_tape* tape, ndvm_dtype dtype, int64_t B, const void* params,
                                           const void* obs, int64_t n_obs, void* loss, void* grad, void* stream) {
  try {
    return host_replay(tape, dtype, B, params, obs, n_obs, loss, grad, stream, false);
  } catch (const std::bad_alloc&) {
    return fail(NDVM_E_OOM, "host allocation failed");
  }
}

ndvm_status ndvm_check_device(const ndvm_tape* tape) {
  ndvm_tape* t = const_cast<ndvm_tape*>(tape);
  if (!t) return fail(NDVM_E_INVALID_ARG, "null tape");
  DevCache* dc = nullptr;
  ndvm_status s = device_cache(t, &dc);
  if (s != NDVM_OK) return s;
  int flag = 0;
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return cuda_fail(e, "synchronize");
  if ((e = cudaMemcpy(&flag, dc->err, sizeof(int), cudaMemcpyDeviceToHost)) != cudaSuccess) return cuda_fail(e, "read flag");
  if (flag) {
    cudaMemset(dc->err, 0, sizeof(int));
    return fail(NDVM_E_DEVICE_CHECK, "a replay kernel met an invalid instruction");
  }
  return NDVM_OK;
}

ndvm_status ndvm_measure_fp64_peak(double* flops_per_s, void* stream) {
  if (!flops_per_s) return fail(NDVM_E_INVALID_ARG, "null output");
  cudaError_t e = measure_fp64_peak(flops_per_s, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "fp64 peak probe");
  return NDVM_OK;
}

ndvm_status ndvm_measure_op_cost(int fn, int iters, double* ns_per_call, void* stream) {
  if (!ns_per_call) return fail(NDVM_E_INVALID_ARG, "null output");
  if (fn < 0 || fn >= NDVM_PROBE_COUNT || iters < 1) return fail(NDVM_E_INVALID_ARG, "unknown probe or iters < 1");
  cudaError_t e = measure_op_cost(fn, iters, ns_per_call, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "function cost probe");
  return NDVM_OK;
}

unsigned long long ndvm_launch_count(void) {
  std::lock_guard<std::mutex> lk(g_launch_mu);
  return g_launches;
}

const char* ndvm_last_error(void) { return g_last_error.c_str(); }

const char* ndvm_version(void) { return "ndvm-gb300 0.1"; }

// Value and gradient without allocating: the workspace is the library's fixed
// scratch array (replay.cu) instead of caller memory, and the tape must already be
// resident on the current device.  No cudaMalloc, cudaFree or other allocating
// call is made here.
ndvm_status ndvm_value_and_grad_noalloc(const ndvm_tape* tape, ndvm_dtype dtype, int64_t B, const void* params,
                                        const void* obs, int64_t n_obs, void* loss, void* grad, void* stream) {
  ndvm_tape* t = const_cast<ndvm_tape*>(tape);
  if (!t) return fail(NDVM_E_INVALID_ARG, "null tape");
  if (dtype != NDVM_F64 && dtype != NDVM_F32) return fail(NDVM_E_INVALID_ARG, "bad dtype");
  if (B < 0) return fail(NDVM_E_INVALID_ARG, "B must be >= 0");
  if (B == 0) return NDVM_OK;
  if (B > (int64_t)1 << 40) return fail(NDVM_E_INVALID_ARG, "B too large");
  const Plan& p = t->grad_plan;
  if (p.n_params > 0 && (!params || !grad)) return fail(NDVM_E_INVALID_ARG, "null params or grad");
  if (!loss) return fail(NDVM_E_INVALID_ARG, "null loss");
  if (n_obs < p.n_obs_min) return fail(NDVM_E_INVALID_ARG, "obs holds fewer values than the program reads");
  if (p.n_obs_min > 0 && !obs) return fail(NDVM_E_INVALID_ARG, "null obs");
  const size_t elem = dtype == NDVM_F32 ? sizeof(float) : sizeof(double);
  const Shape sh = launch_shape(p, elem, B);
  const int tpb = sh.tpb, log2g = sh.log2g;
  const size_t smem = sh.smem;
  if (smem > kSmemLimit) return fail(NDVM_E_UNSUPPORTED, "tape needs more slots per lane than shared memory holds");
  const int lanes_per_block = tpb >> log2g;
  // the scratch holds the shared per-point values first, then the per-lane saves
  const size_t der_bytes = derived_bytes(p, elem);
  const size_t lane_scratch = der_bytes <= kNoAllocScratchBytes ? kNoAllocScratchBytes - der_bytes : 0;
  int64_t chunk = B;
  if (der_bytes > kNoAllocScratchBytes)
    return fail(NDVM_E_INVALID_ARG, "this tape's extended observations need " + std::to_string(der_bytes) +
                                        " bytes; the fixed scratch holds " + std::to_string(kNoAllocScratchBytes) + " bytes");
  if (p.n_save > 0) {
    const size_t per_lane = (size_t)p.n_save * elem;
    const size_t per_block = per_lane * sh.chunk_lanes;
    if (per_block > lane_scratch)
      return fail(NDVM_E_INVALID_ARG, "this tape needs " + std::to_string(per_block) + " bytes of workspace per block of " +
                                          std::to_string(sh.chunk_lanes) + " lanes; the fixed scratch holds " +
                                          std::to_string(kNoAllocScratchBytes) + " bytes");
    int64_t fit = (int64_t)(lane_scratch / per_lane);
    if (fit < B) chunk = fit - fit % sh.chunk_lanes;
  }
  // one launch covers at most kMaxChunk lanes, so its grid stays far below 2^31 blocks
  if (chunk > kMaxChunk) chunk = kMaxChunk - kMaxChunk % sh.chunk_lanes;
  if ((chunk + lanes_per_block - 1) / lanes_per_block > 0x7fffffff)
    return fail(NDVM_E_INVALID_ARG, "too many lanes for one launch");
  DevCache* dc = nullptr;
  {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    std::lock_guard<std::mutex> lk(t->mu);
    auto it = t->dev.find(dev);
    if (it == t->dev.end())
      return fail(NDVM_E_INVALID_ARG, "tape is not resident on this device; one ndvm_forward or ndvm_value_and_grad "
                                      "call uploads it (that call allocates)");
    dc = &it->second;
  }
  void* scratch = nullptr;
  cudaError_t e = noalloc_scratch(&scratch);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress");
  if (der_bytes > 0) {
    ndvm_status s = run_derive(p, dc->grad, dtype, obs, scratch, !reads_both(sh), dc->err, stream);
    if (s != NDVM_OK) return s;
  }
  ReplayArgs a;
  plan_args(a, p, dc->grad, sh, dtype, dc->err);
  set_obs(a, sh, obs, der_bytes > 0 ? scratch : nullptr);
  a.params = params;
  a.loss = loss;
  a.grad = grad;
  a.save = static_cast<char*>(scratch) + der_bytes;
  a.save_ld = chunk;
  for (int64_t l0 = 0; l0 < B; l0 += chunk) {
    a.lane0 = l0;
    a.lane_end = l0 + chunk < B ? l0 + chunk : B;
    const int64_t blocks = (a.lane_end - l0 + lanes_per_block - 1) / lanes_per_block;
    {
      std::lock_guard<std::mutex> lk(g_launch_mu);
      e = launch_replay(a, dtype == NDVM_F32, (int)blocks, tpb, smem, (cudaStream_t)stream);
      g_launches++;
    }
    if (e != cudaSuccess) return cuda_fail(e, "replay launch");
  }
  return NDVM_OK;
}

}  // extern "C"
