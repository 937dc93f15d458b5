// Batched stepping of many independent periodic fields (the C-ABI lbch_batch_*),
// included at the end of lbch_api.cu so that it shares the context machinery.
//
// One kernel launch advances every field of the batch by one time step. Each warp
// reads its (field, strip, segment) from a task table and its field's geometry from
// a field table, then runs the same warp body as the single-field kernel, so every
// node is computed exactly as it would be alone. Kernel boundaries separate the time
// steps: there is no grid-wide barrier and no spin-wait. Steps are replayed from CUDA
// graphs of BATCH_GRAPH_STEPS steps to amortise launch cost. At creation a small
// autotuner times candidate row-segment lengths on the zeroed buffers and keeps the
// fastest: long ones (less warm-up) where the batch fills the GPU, short ones where a
// step is one walk of a segment.
#pragma once

#include <algorithm>
#include <vector>

namespace lbch {

constexpr int BATCH_GRAPH_STEPS = 64;                             // launches per CUDA graph (even)
// Rows per warp tried by the tuner. 64 steps of 16 fields of 64^2 to 200^2: 2136 us with 32 rows at
// least, 711 with 4 (a step was one walk of 32 rows and its warm-up); of 256 fields 6418 and 4005.
constexpr int BATCH_ROW_TARGETS[] = {4, 8, 16, 32, 64, 128, 256, 512, 1024};
constexpr int N_ROW_TARGETS = sizeof(BATCH_ROW_TARGETS) / sizeof(int);

template <int ST, bool VEC, int RT, bool MI, bool MO>
__global__ void __launch_bounds__(STEP_WARPS * 32, (Pipe<ST, VEC, MI>::MIN_CTAS))
    step_batch_kernel(const __grid_constant__ StepArgs a, const Field* __restrict__ fields,
                      const int4* __restrict__ tasks, int n_tasks, int parity) {
  extern __shared__ float4 smem_slots[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int warp = blockIdx.x * STEP_WARPS + wib;
  if (warp >= n_tasks) return;  // whole warps only (tasks: those of the launch's group)
  const int4 t = tasks[warp];   // field, strip, segment
  Field fd = fields[t.x];
  if (parity) {
    const Buf tmp = fd.src;
    fd.src = fd.dst;
    fd.dst = tmp;
  }
  float4* slots = smem_slots + wib * (Pipe<ST, VEC, MI>::SLOTS * Pipe<ST, VEC, MI>::SLOT_F4);
  launch_warp<ST, VEC, RT, MI, MO>(a, fd, t.y, t.z, slots, lane);
}

}  // namespace lbch

// The fields that one launch steps together: all those of one collision form. FP32 fields that
// step in R_SUMS and moment form alone do so here, apart from the others; the two groups' runs
// have nothing in common and go on two streams.
struct BatchGroup {
  int first;             // first task
  int n_tasks;
  int rates;             // R_*
  bool vec;              // every field of the group has 16-byte rows
  bool mform;            // runs of steps go through moment form
  int cur;               // buffer of the group's current state
  cudaGraphExec_t graph; // BATCH_GRAPH_STEPS steps from buffer 0
};

struct lbch_batch {
  int count;
  std::vector<lbch_ctx*> fields;  // one context per field, sharing the scratch area
  std::vector<long long> nodes;
  std::vector<int> group_of;     // each field's group
  lbch_params common;
  cudaStream_t stream;
  cudaStream_t side;             // private stream: captures the graphs, runs the second of two groups
  cudaEvent_t fork, join;        // a run of two groups: from the caller's stream to side and back
  StepArgs sa;
  BatchGroup group[2];           // fields in R_SUMS, and the others (either may be empty)
  Field* d_fields;               // field table (parity 0 buffers), device
  int4* d_tasks;                 // task table, device
  size_t max_tasks;
  int rows_target;               // chosen by the tuner
  float tune_ms[N_ROW_TARGETS];
  int64_t steps;
  bool failed;
  char err[512];
};

namespace {

void batch_err(lbch_batch* b, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(b->err, sizeof(b->err), fmt, ap);
  va_end(ap);
}

bool batch_cuda_failed(lbch_batch* b, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return false;
  b->failed = true;
  batch_err(b, "%s: %s", what, cudaGetErrorString(e));
  return true;
}

// Parameters of field i: the common ones with this field's size and anisotropy.
lbch_params field_params(const lbch_params* common, int32_t nx, int32_t ny, double alpha) {
  lbch_params p = *common;
  p.nx = nx;
  p.ny = ny;
  p.alpha = alpha;
  return p;
}

int n_strips_of(int nx) { return n_strips_for(nx); }

// Rows of a field's segments for a rows-per-warp target: as even as whole rows allow.
int segment_rows(int ny, int rows) {
  const int segs = std::max(1, (ny + rows - 1) / rows);
  return (ny + segs - 1) / segs;
}

// Task list for a rows-per-warp target: the fields of group 0 first, in a group the largest
// fields first (longest work first), and within a field the strips of a segment next to each
// other (they share halos). Returns the number of group 0's tasks.
int build_tasks(const int32_t* nx, const int32_t* ny, int count, int rows, const std::vector<int>& group_of,
                std::vector<int4>& tasks, std::vector<int>& seg_len) {
  std::vector<int> order(count);
  for (int i = 0; i < count; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    if (group_of[x] != group_of[y]) return group_of[x] < group_of[y];
    return (long long)nx[x] * ny[x] > (long long)nx[y] * ny[y];
  });
  tasks.clear();
  seg_len.assign(count, 1);
  int first_group = 0;
  for (int f : order) {
    const int len = segment_rows(ny[f], rows);
    seg_len[f] = len;
    const int nseg = (ny[f] + len - 1) / len;
    for (int g = 0; g < nseg; ++g)
      for (int s = 0; s < n_strips_of(nx[f]); ++s) tasks.push_back(make_int4(f, s, g, 0));
    if (group_of[f] == 0) first_group = (int)tasks.size();
  }
  return first_group;
}

size_t max_task_count(const int32_t* nx, const int32_t* ny, int count) {
  size_t m = 0;
  for (const int rows : BATCH_ROW_TARGETS) {
    size_t n = 0;
    for (int f = 0; f < count; ++f) {
      const int len = segment_rows(ny[f], rows);
      n += (size_t)((ny[f] + len - 1) / len) * n_strips_of(nx[f]);
    }
    m = std::max(m, n);
  }
  return m;
}

const char* check_batch(const lbch_params* common, int32_t count, const int32_t* nx, const int32_t* ny,
                        const double* alpha) {
  if (!common || !nx || !ny || count < 1 || count > (1 << 20)) return "bad batch arguments";
  for (int i = 0; i < count; ++i) {
    const lbch_params p = field_params(common, nx[i], ny[i], alpha ? alpha[i] : common->alpha);
    if (const char* e = check_params(&p)) return e;
  }
  return nullptr;
}

template <int ST, bool VEC, int RT, bool MI, bool MO>
struct BatchK {
  static constexpr int SMEM = step_smem<ST, VEC, MI>();
  static cudaError_t configure() {
    return cudaFuncSetAttribute(step_batch_kernel<ST, VEC, RT, MI, MO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                SMEM);
  }
  static void launch(const lbch_batch* b, const BatchGroup& g, cudaStream_t s, int parity) {
    const int blocks = (g.n_tasks + STEP_WARPS - 1) / STEP_WARPS;
    launch_dep(step_batch_kernel<ST, VEC, RT, MI, MO>, blocks, STEP_WARPS * 32, SMEM, s, b->sa, b->d_fields,
               b->d_tasks + g.first, g.n_tasks, parity);
  }
};

// The batch kernel with the template arguments of a single-field instantiation.
template <int ST, bool VEC, int RT, bool MI, bool MO>
BatchK<ST, VEC, RT, MI, MO> batch_kernel_of(StepK<ST, VEC, RT, MI, MO>) { return {}; }

cudaError_t configure_batch_kernel(const lbch_batch* b, const BatchGroup& g, int form) {
  cudaError_t e = cudaSuccess;
  with_step_kernel(b->common.storage, g.vec, g.rates, form, [&](auto k) { e = batch_kernel_of(k).configure(); });
  return e;
}

void batch_launch(const lbch_batch* b, const BatchGroup& g, cudaStream_t s, int parity, int form) {
  with_step_kernel(b->common.storage, g.vec, g.rates, form,
                   [&](auto k) { batch_kernel_of(k).launch(b, g, s, parity); });
}
int run_form(const BatchGroup& g) { return g.mform ? MOM_MOM : POP_POP; }

// A run of two groups: group 1 goes on the side stream, from the caller's stream and back to it.
bool two_groups(const lbch_batch* b) { return b->group[0].n_tasks && b->group[1].n_tasks; }
cudaStream_t stream_of(const lbch_batch* b, const BatchGroup& g) {
  return two_groups(b) && &g == &b->group[1] ? b->side : b->stream;
}
lbch_status batch_fork(lbch_batch* b) {
  if (two_groups(b) && (batch_cuda_failed(b, cudaEventRecord(b->fork, b->stream), "step: fork") ||
                        batch_cuda_failed(b, cudaStreamWaitEvent(b->side, b->fork, 0), "step: fork")))
    return LBCH_ECUDA;
  return LBCH_OK;
}
lbch_status batch_join(lbch_batch* b) {
  if (two_groups(b) && (batch_cuda_failed(b, cudaEventRecord(b->join, b->side), "step: join") ||
                        batch_cuda_failed(b, cudaStreamWaitEvent(b->stream, b->join, 0), "step: join")))
    return LBCH_ECUDA;
  return LBCH_OK;
}

// Uploads a task list for `rows` and sets the per-field segment lengths in the field table.
lbch_status batch_use_rows(lbch_batch* b, const int32_t* nx, const int32_t* ny, int rows) {
  std::vector<int4> tasks;
  std::vector<int> seg_len;
  const int first_group = build_tasks(nx, ny, b->count, rows, b->group_of, tasks, seg_len);
  std::vector<Field> table(b->count);
  for (int i = 0; i < b->count; ++i) {
    Field f = b->fields[i]->fld;
    f.seg_len = seg_len[i];
    f.src = b->fields[i]->buf[0];
    f.dst = b->fields[i]->buf[1];
    table[i] = f;
  }
  if (batch_cuda_failed(b, cudaMemcpyAsync(b->d_tasks, tasks.data(), tasks.size() * sizeof(int4),
                                           cudaMemcpyHostToDevice, b->stream), "batch: upload tasks") ||
      batch_cuda_failed(b, cudaMemcpyAsync(b->d_fields, table.data(), table.size() * sizeof(Field),
                                           cudaMemcpyHostToDevice, b->stream), "batch: upload fields") ||
      batch_cuda_failed(b, cudaStreamSynchronize(b->stream), "batch: upload sync"))
    return LBCH_ECUDA;
  b->group[0].first = 0;
  b->group[0].n_tasks = first_group;
  b->group[1].first = first_group;
  b->group[1].n_tasks = (int)tasks.size() - first_group;
  b->rows_target = rows;
  return LBCH_OK;
}

}  // namespace

extern "C" {

size_t lbch_batch_workspace_bytes(const lbch_params* common, int32_t count, const int32_t* nx, const int32_t* ny) {
  if (check_batch(common, count, nx, ny, nullptr)) return 0;
  size_t total = 0, scratch = 0;
  for (int i = 0; i < count; ++i) {
    const lbch_params p = field_params(common, nx[i], ny[i], common->alpha);
    total += 2 * state_bytes(&p);
    scratch = std::max(scratch, scratch_bytes(&p));
  }
  return total + scratch + align_up((size_t)count * sizeof(Field)) +
         align_up(max_task_count(nx, ny, count) * sizeof(int4));
}

lbch_status lbch_batch_create(const lbch_params* common, int32_t count, const int32_t* nx, const int32_t* ny,
                              const double* alpha, void* d_workspace, size_t bytes, void* cuda_stream,
                              lbch_batch** out) {
  if (!out || check_batch(common, count, nx, ny, alpha)) return LBCH_EINVAL;
  const size_t need = lbch_batch_workspace_bytes(common, count, nx, ny);
  if (!d_workspace || bytes < need || ((uintptr_t)d_workspace % ALIGN) != 0) return LBCH_ENOMEM;
  lbch_batch* b = new (std::nothrow) lbch_batch();
  if (!b) return LBCH_ENOMEM;
  b->count = count;
  b->common = *common;
  b->stream = (cudaStream_t)cuda_stream;
  b->side = nullptr;
  b->fork = b->join = nullptr;
  b->group[0] = b->group[1] = BatchGroup{};
  b->steps = 0;
  b->failed = false;
  b->err[0] = 0;
  // Layout: field states, shared scratch, field table, task table.
  char* q = (char*)d_workspace;
  size_t scratch = 0;
  for (int i = 0; i < count; ++i) {
    const lbch_params p = field_params(common, nx[i], ny[i], alpha ? alpha[i] : common->alpha);
    scratch = std::max(scratch, scratch_bytes(&p));
  }
  char* states = q;
  size_t state_total = 0;
  for (int i = 0; i < count; ++i) {
    const lbch_params p = field_params(common, nx[i], ny[i], common->alpha);
    state_total += 2 * state_bytes(&p);
  }
  char* shared_scratch = states + state_total;
  b->d_fields = (Field*)(shared_scratch + scratch);
  b->d_tasks = (int4*)((char*)b->d_fields + align_up((size_t)count * sizeof(Field)));
  b->max_tasks = max_task_count(nx, ny, count);
  b->fields.assign(count, nullptr);
  b->nodes.assign(count, 0);
  char* st = states;
  for (int i = 0; i < count; ++i) {
    const lbch_params p = field_params(common, nx[i], ny[i], alpha ? alpha[i] : common->alpha);
    lbch_status r = ctx_setup(&p, st, shared_scratch, b->stream, &b->fields[i]);
    if (r != LBCH_OK) {
      lbch_batch_destroy(b);
      return r;
    }
    st += 2 * state_bytes(&p);
    b->nodes[i] = (long long)nx[i] * ny[i];
  }
  b->sa = b->fields[0]->sa;  // the same scheme constants for every field
  // Group 0: FP32 fields in R_SUMS. The 16-bit storages step in moment form where every field of
  // the batch has 16-byte rows (a ragged field puts the group on the scalar kernels).
  b->group_of.assign(count, 1);
  for (int i = 0; i < count; ++i)
    if (b->fields[i]->rates == R_SUMS) b->group_of[i] = 0;
  b->group[0].rates = R_SUMS;
  b->group[0].vec = b->group[1].vec = true;
  b->group[0].mform = true;
  b->group[1].mform = common->storage != LBCH_STORE_F32;
  for (int i = 0; i < count; ++i) {
    const lbch_ctx* c = b->fields[i];
    BatchGroup& g = b->group[b->group_of[i]];
    if (c->rates != R_SUMS) g.rates = c->rates;
    g.vec = g.vec && c->vec;
    g.mform = g.mform && c->mform;
  }
  bool used[2] = {false, false};
  for (int g : b->group_of) used[g] = true;
  cudaError_t e = cudaSuccess;
  for (int g = 0; g < 2; ++g)
    for (int form = POP_POP; used[g] && e == cudaSuccess && form <= (b->group[g].mform ? MOM_MOM : POP_POP); ++form)
      e = configure_batch_kernel(b, b->group[g], form);
  if (batch_cuda_failed(b, e, "batch: configure") ||
      batch_cuda_failed(b, cudaStreamCreateWithFlags(&b->side, cudaStreamNonBlocking), "batch: stream") ||
      batch_cuda_failed(b, cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming), "batch: event") ||
      batch_cuda_failed(b, cudaEventCreateWithFlags(&b->join, cudaEventDisableTiming), "batch: event")) {
    lbch_batch_destroy(b);
    return LBCH_ECUDA;
  }
  // Autotune the row-segment length on zeroed buffers (the kernel's work does not depend on the
  // values), the groups on their streams as a run has them, then capture the graphs for the winner.
  cudaEvent_t t0 = nullptr, t1 = nullptr;
  bool ok = !batch_cuda_failed(b, cudaMemsetAsync(states, 0, state_total, b->stream), "batch: clear") &&
            !batch_cuda_failed(b, cudaEventCreate(&t0), "batch: event") &&
            !batch_cuda_failed(b, cudaEventCreate(&t1), "batch: event");
  auto time_steps = [&](int n, float& ms) {  // n steps of every field; false on an error
    cudaEventRecord(t0, b->stream);
    if (batch_fork(b) != LBCH_OK) return false;
    for (const BatchGroup& g : b->group)
      for (int k = 0; g.n_tasks && k < n; ++k) batch_launch(b, g, stream_of(b, g), k & 1, run_form(g));
    if (batch_join(b) != LBCH_OK) return false;
    cudaEventRecord(t1, b->stream);
    if (batch_cuda_failed(b, cudaEventSynchronize(t1), "batch: tune")) return false;
    float t = 0.0f;
    cudaEventElapsedTime(&t, t0, t1);
    ms += t;
    return true;
  };
  // Longest segments first. A target that splits every field as the one before is the same run, and
  // one whose first two steps took an eighth longer than the best one's did is not timed further (the
  // 512-field sweep: 59 ms of creation with eight launches for each of nine targets, 35 this way).
  int best = -1;
  float best_two = 0.0f;
  for (int r = N_ROW_TARGETS - 1; ok && r >= 0; --r) {
    bool same = r < N_ROW_TARGETS - 1;
    for (int i = 0; same && i < count; ++i)
      same = segment_rows(ny[i], BATCH_ROW_TARGETS[r]) == segment_rows(ny[i], BATCH_ROW_TARGETS[r + 1]);
    if (same) {
      b->tune_ms[r] = b->tune_ms[r + 1];
      continue;
    }
    float warm = 0.0f, ms = 0.0f;
    ok = batch_use_rows(b, nx, ny, BATCH_ROW_TARGETS[r]) == LBCH_OK && time_steps(1, warm) && time_steps(2, ms);
    b->tune_ms[r] = ms / 2.0f;
    if (!ok || (best >= 0 && ms > 1.125f * best_two)) continue;
    const float two = ms;
    ok = time_steps(4, ms);
    b->tune_ms[r] = ms / 6.0f;
    if (best >= 0 && b->tune_ms[r] >= b->tune_ms[best]) continue;
    best = r;
    best_two = two;
  }
  if (t0) cudaEventDestroy(t0);
  if (t1) cudaEventDestroy(t1);
  if (ok && b->rows_target != BATCH_ROW_TARGETS[best]) ok = batch_use_rows(b, nx, ny, BATCH_ROW_TARGETS[best]) == LBCH_OK;
  for (BatchGroup& gr : b->group) {
    if (!ok || !gr.n_tasks) continue;
    cudaGraph_t g = nullptr;
    ok = !batch_cuda_failed(b, cudaStreamBeginCapture(b->side, cudaStreamCaptureModeThreadLocal),
                            "batch: capture");
    if (ok) {
      for (int k = 0; k < BATCH_GRAPH_STEPS; ++k) batch_launch(b, gr, b->side, k & 1, run_form(gr));
      ok = !batch_cuda_failed(b, cudaStreamEndCapture(b->side, &g), "batch: capture end");
    }
    if (ok) ok = !batch_cuda_failed(b, cudaGraphInstantiate(&gr.graph, g, 0), "batch: instantiate");
    if (g) cudaGraphDestroy(g);
  }
  if (!ok) {
    lbch_batch_destroy(b);
    return LBCH_ECUDA;
  }
  *out = b;
  return LBCH_OK;
}

lbch_status lbch_batch_init_field(lbch_batch* b, int32_t i, const double* h_phi0) {
  if (!b || i < 0 || i >= b->count) return LBCH_EINVAL;
  if (b->failed) return LBCH_ESTATE;
  lbch_ctx* c = b->fields[i];
  if (b->steps % 2 != 0) {
    batch_err(b, "init_field: initialise fields before the first step or after an even number of steps");
    return LBCH_EINVAL;
  }
  // Into the buffer of the field's group (a run in moment form may leave it on buffer 1):
  // lbch_init_field writes what the context calls buffer 0.
  const int cur = b->group[b->group_of[i]].cur;
  if (cur) std::swap(c->buf[0], c->buf[1]);
  lbch_status st = lbch_init_field(c, h_phi0);
  if (cur) {
    std::swap(c->buf[0], c->buf[1]);
    c->cur = 1;
  }
  if (st != LBCH_OK) batch_err(b, "field %d: %s", i, lbch_last_error(c));
  if (st == LBCH_ECUDA) b->failed = true;
  return st;
}

lbch_status lbch_batch_step(lbch_batch* b, int64_t n) {
  if (!b || n < 0) return LBCH_EINVAL;
  if (b->failed) return LBCH_ESTATE;
  for (lbch_ctx* c : b->fields)
    if (!c->has_state) {
      batch_err(b, "step: every field needs lbch_batch_init_field first");
      return LBCH_EINVAL;
    }
  if (n > 0 && batch_fork(b) != LBCH_OK) return LBCH_ECUDA;
  for (BatchGroup& g : b->group) {
    if (!g.n_tasks) continue;
    const cudaStream_t s = stream_of(b, g);
    int64_t left = n;
    auto one = [&](int form) {
      batch_launch(b, g, s, g.cur, form);
      g.cur ^= 1;
    };
    // Gather, steps in moment form, and a last one back to populations.
    const bool mom = g.mform && n >= MOM_MIN_STEPS;
    const int form = mom ? MOM_MOM : POP_POP;
    if (mom) {
      one(POP_MOM);
      --left;  // the last step
    }
    if (form == run_form(g) && left >= BATCH_GRAPH_STEPS + (g.cur ? 1 : 0) && !capturing(s)) {
      if (g.cur == 1) {  // back to parity 0, where the graph starts
        one(form);
        --left;
      }
      for (; left >= BATCH_GRAPH_STEPS; left -= BATCH_GRAPH_STEPS)
        if (batch_cuda_failed(b, cudaGraphLaunch(g.graph, s), "step: graph launch")) return LBCH_ECUDA;
    }
    for (; left > 0; --left) one(form);
    if (mom) one(MOM_POP);
  }
  if (n > 0 && batch_join(b) != LBCH_OK) return LBCH_ECUDA;
  b->steps += n;
  for (int i = 0; i < b->count; ++i) {
    b->fields[i]->cur = b->group[b->group_of[i]].cur;
    b->fields[i]->steps = b->steps;
  }
  if (batch_cuda_failed(b, cudaGetLastError(), "step: launch")) return LBCH_ECUDA;
  return LBCH_OK;
}

#define LBCH_BATCH_FIELD_CALL(NAME, CALL)                              \
  lbch_status NAME {                                                   \
    if (!b || i < 0 || i >= b->count) return LBCH_EINVAL;             \
    if (b->failed) return LBCH_ESTATE;                                 \
    lbch_ctx* c = b->fields[i];                                        \
    lbch_status st = CALL;                                             \
    if (st != LBCH_OK) batch_err(b, "field %d: %s", i, lbch_last_error(c)); \
    if (st == LBCH_ECUDA) b->failed = true;                            \
    return st;                                                         \
  }

LBCH_BATCH_FIELD_CALL(lbch_batch_get_field(lbch_batch* b, int32_t i, double* h_phi), lbch_get_field(c, h_phi))
LBCH_BATCH_FIELD_CALL(lbch_batch_get_phi_device(lbch_batch* b, int32_t i, float* d_phi), lbch_get_phi_device(c, d_phi))
LBCH_BATCH_FIELD_CALL(lbch_batch_mass(lbch_batch* b, int32_t i, double* out), lbch_mass(c, out))
LBCH_BATCH_FIELD_CALL(lbch_batch_free_energy(lbch_batch* b, int32_t i, double* out), lbch_free_energy(c, out))
#undef LBCH_BATCH_FIELD_CALL

int32_t lbch_batch_rows_target(const lbch_batch* b) { return b ? b->rows_target : -1; }

int64_t lbch_batch_steps_taken(const lbch_batch* b) { return b ? b->steps : -1; }

const char* lbch_batch_last_error(const lbch_batch* b) { return b ? b->err : "batch is NULL"; }

void lbch_batch_destroy(lbch_batch* b) {
  if (!b) return;
  for (BatchGroup& g : b->group)
    if (g.graph) cudaGraphExecDestroy(g.graph);
  if (b->fork) cudaEventDestroy(b->fork);
  if (b->join) cudaEventDestroy(b->join);
  if (b->side) cudaStreamDestroy(b->side);
  for (lbch_ctx* c : b->fields) delete c;
  delete b;
}

}  // extern "C"
