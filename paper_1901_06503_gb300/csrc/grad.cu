// grad.cu -- the differentiated forward operator: g = P W(c) h with
// wavefield checkpoints, and the backward pass giving grad_h = A^T grad_g and
// grad_c = d<grad_g, A(c) h>/dc (dt held fixed: Nt is piecewise constant in c).
//
// Forward: the three-term leapfrog of the wave model (Sec. 2.1) saves the
// pair (p^{sk}, p^{sk+1}) every k steps.  Backward: the transposed recurrence
// runs from lambda^{Nt} = P^T grad_g down to lambda^0 = grad_h; written for
// mu = (kappa/12) lambda it is the forward three-term step again
// (mu^n = 2 mu^{n+1} - mu^{n+2} + kappa L mu^{n+1}).  Segment by segment, from
// the last, the states p^n of the segment are recomputed from its checkpoint
// and the kappa-derivatives mu^{n+1} L(p^n) (weight 1/2 for the start step)
// are accumulated; grad_c = 2 acc / c because dkappa/dc = 2 kappa / c and the
// factors kappa/12 and 12 cancel.  Memory: 2 ceil(Nt/k) + k + 2 volumes (on small
// grids up to k more, with which the segments overlap).
//
// Where the resident time loop runs (FP32, N <= 128), the forward pass is one
// cooperative launch that stores the checkpoints as it goes, and a segment of
// the backward pass two: recompute (writing L(p^n) in place of p^n) and
// transposed steps with the accumulation; up to N = 84 the transposed steps of a
// segment and the recompute of the one before share a launch.  Elsewhere they are loops of launches.
// FP32 volumes with ragged rows run on padded rows (wave_plan), FP64 ones as
// they are.
#include "internal.cuh"

namespace ffpat {
namespace {

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct Ckpt {
  size_t vol = 0;
  int nseg = 0, every = 0, nvol = 0;  // nvol: segment volumes
  bool paired = false;                // room for two segments' volumes
  unsigned char* base = nullptr;
  void* a(int s) const { return base + (size_t)(2 * s) * vol; }
  void* b(int s) const { return base + (size_t)(2 * s + 1) * vol; }
  void* seg(int j) const { return base + (size_t)(2 * nseg + j) * vol; }  // j < nvol
  void* acc() const { return base + (size_t)(2 * nseg + nvol) * vol; }
  size_t bytes() const { return (size_t)(2 * nseg + nvol + 1) * vol; }
};

// (have: bytes at base)
int ckpt_layout(const Plan& pl, int nt, int every, void* base, size_t have, Ckpt* ck) {
  if (pl.pad != 0) return report(FFPAT_EINVAL, "the differentiated operator needs pad = 0");
  if (every < 1 || every > 4096) return report(FFPAT_EINVAL, "checkpoint interval %d", every);
  // (FP32 volumes may have padded rows, FP64 ones never: see grad_view)
  const size_t row = pl.esize == 4 ? padded_row(pl) : pl.n;
  ck->vol = up256((size_t)pl.n * pl.n * row * pl.esize);
  ck->every = every;
  ck->nseg = (nt + every - 1) / every;
  ck->nvol = every + 1;
  ck->base = (unsigned char*)base;
  // FP32 on small grids: room for two segments at a time, where there are two and
  // the buffer holds them (see the resident branch of the backward pass)
  if (pl.esize == 4 && pl.n <= kSegmentPairMaxN && ck->nseg >= 2) {
    Ckpt two = *ck;
    two.nvol += ck->nseg > 2 ? every : nt - every;  // the odd segments' volumes
    two.paired = true;
    if (two.bytes() <= have) *ck = two;
  }
  if (ck->bytes() > have)
    return report(FFPAT_ENOMEM, "checkpoint buffer %zu < %zu bytes", have, ck->bytes());
  return FFPAT_OK;
}

// the three-term stepper runs this path for every precision (FP32-Kahan
// problems take FP32 three-term steps: the same discrete operator)
void as_three_term(Plan& pl) {
  if (pl.prec == FFPAT_FP32_KAHAN) pl.prec = FFPAT_FP32;
}

bool use_tma(const Plan& pl, const Ckpt& ck, const void* a) {
  const void* ptrs[8] = {a, pl.kap, pl.s[0], pl.s[1], pl.s[2], pl.s[3], pl.x, ck.base};
  return tma_supported(pl, ptrs, 8) && (ck.vol % 16) == 0;
}

// The rows the steps run on: padded in FP32; dense in FP64 (whose accumulation
// kernel is the plain one) and for a checkpoint buffer that TMA cannot address.  The
// same for the forward and the backward pass.
Rows grad_rows(const ffpat_problem* pr, const void* ckpt) {
  const bool tma = pr && pr->precision != FFPAT_FP64 && ((uintptr_t)ckpt & 15) == 0;
  return tma ? Rows::kPadded : Rows::kDense;
}

// two steps per pass in the checkpointed loops: W's rule, and checkpoints at
// even steps (the passes advance the pair (p^m, p^{m+1}) by two)
bool use_two(const Plan& pl, const Ckpt& ck, bool tma) {
  return two_step_three_term(pl, tma) && ck.every % 2 == 0 && pl.s[2] && pl.s[3];
}

}  // namespace
}  // namespace ffpat

using namespace ffpat;

extern "C" {

size_t ffpat_ckpt_bytes(const ffpat_problem* problem, int32_t nt, int32_t every) {
  Plan pl;
  if (ffpat_workspace_bytes(problem) == 0 || nt < 1) return 0;
  if (attach(problem, pl, (void*)256, ffpat_workspace_bytes(problem)) != FFPAT_OK) return 0;
  Ckpt ck;
  if (ckpt_layout(pl, nt, every, nullptr, (size_t)-1, &ck) != FFPAT_OK) return 0;
  return ck.bytes();
}

int ffpat_forward_ckpt(const ffpat_problem* problem, const void* c, const void* h, void* g,
                       int32_t every, void* ckpt, size_t ckpt_bytes, void* ws, size_t ws_bytes,
                       void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  Plan pl;
  const int rc0 = setup(problem, pl, c, ws, ws_bytes, st, grad_rows(problem, ckpt));
  if (rc0 != FFPAT_OK) return rc0;
  if (!h || !g || !ckpt) return report(FFPAT_EINVAL, "h, g or ckpt is NULL");
  as_three_term(pl);
  Ckpt ck;
  const int rc1 = ckpt_layout(pl, pl.nt, every, ckpt, ckpt_bytes, &ck);
  if (rc1 != FFPAT_OK) return rc1;
  const Plan w = wave_plan(pl);
  const void* in = h;
  if (w.np != w.n) {  // the source in padded rows
    const int rc = launch_embed(pl, h, pl.xw, st);
    if (rc != FFPAT_OK) return rc;
    in = pl.xw;
  }
  const bool tma = use_tma(w, ck, in);
  if (resident_segments(w, tma, st)) {
    const ResidentSave save{ck.base, ck.vol / 4, every};
    const void* last = nullptr;
    bool refused = false;
    const int rc = launch_wave_resident(w, 0, in, nullptr, pl.s[0], pl.s[1], &last, st, &refused,
                                        &save);
    if (rc == FFPAT_OK)
      return launch_project(w, last, g, nullptr, st, nullptr, project_scratch(pl, last));
    if (!refused) return rc;  // refused: step by step
  }
  const bool two = use_two(w, ck, tma);
  // S[a] = p^m, S[b] = p^{m+1}; a two-step pass writes the other pair
  void* S[4] = {pl.s[0], pl.s[1], pl.s[2], pl.s[3]};
  int a = 0, b = 1;
  int rc = step3(w, tma, true, in, nullptr, S[b], S[a], st);  // p^0, p^1
  if (rc != FFPAT_OK) return rc;
  const size_t vb = (size_t)w.n * w.n * w.np * w.esize;
  if (cudaMemcpyAsync(ck.a(0), S[a], vb, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
      cudaMemcpyAsync(ck.b(0), S[b], vb, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return check_launch("checkpoint copy");
  for (int m = 0; m + 1 < pl.nt;) {
    if (two && m + 3 <= pl.nt) {
      rc = launch_step2_f32(w, S[a], S[b], S[a ^ 2], S[b ^ 2], st);  // p^{m+2}, p^{m+3}
      a ^= 2;
      b ^= 2;
      m += 2;
    } else {
      rc = step3(w, tma, false, S[b], S[a], S[a], nullptr, st);  // p^{m+2} over p^m
      const int t = a;
      a = b;
      b = t;
      m += 1;
    }
    if (rc != FFPAT_OK) return rc;
    if (m % every == 0) {
      const int s = m / every;
      if (cudaMemcpyAsync(ck.a(s), S[a], vb, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
          cudaMemcpyAsync(ck.b(s), S[b], vb, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return check_launch("checkpoint copy");
    }
  }
  return launch_project(w, S[b], g, nullptr, st, nullptr, project_scratch(pl, S[b]));
}

int ffpat_backward(const ffpat_problem* problem, const void* c, const void* grad_g, void* grad_h,
                   void* grad_c, int32_t every, void* ckpt, size_t ckpt_bytes, void* ws,
                   size_t ws_bytes, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  Plan pl;
  const int rc0 = setup(problem, pl, c, ws, ws_bytes, st, grad_rows(problem, ckpt));
  if (rc0 != FFPAT_OK) return rc0;
  if (!grad_g || !ckpt) return report(FFPAT_EINVAL, "grad_g or ckpt is NULL");
  as_three_term(pl);
  Ckpt ck;
  const int rc1 = ckpt_layout(pl, pl.nt, every, ckpt, ckpt_bytes, &ck);
  if (rc1 != FFPAT_OK) return rc1;
  const Plan w = wave_plan(pl);
  const bool tma = use_tma(w, ck, nullptr);
  const bool two = use_two(w, ck, tma);
  bool resident = resident_segments(w, tma, st);  // until a launch is turned down
  const size_t vb = (size_t)w.n * w.n * w.np * w.esize;
  // mu^{Nt} = (kappa / 12) P^T grad_g, mu^{Nt+1} = 0
  // B[u] = mu^{n+1}, B[v] = mu^{n+2}; a pass writes into the other two buffers
  void* B[4] = {pl.x, pl.s[0], pl.s[1], pl.s[2]};
  const bool two_t = two_step_three_term(w, tma) && pl.s[1] && pl.s[2];
  int u = 0, v = 1;
  auto others = [&](int* x, int* y) {
    *x = 0;
    while (*x == u || *x == v) ++*x;
    *y = *x + 1;
    while (*y == u || *y == v) ++*y;
  };
  const void* end = nullptr;  // start(mu^1) - mu^2 where a resident segment left it
  const void* tmp = nullptr;  // start(mu^1) else
  int rc = launch_backproject(w, grad_g, B[u], w.kap, st, backproject_scratch(pl, grad_g));
  if (rc != FFPAT_OK) return rc;
  if (cudaMemsetAsync(B[v], 0, vb, st) != cudaSuccess ||
      cudaMemsetAsync(ck.acc(), 0, vb, st) != cudaSuccess)
    return check_launch("backward init");
  // resident segments: L(p^{lo+j}) in the segment volumes (two sets where the
  // recompute of a segment runs beside the transposed steps of the next), the
  // recomputed states through two spare volumes
  const bool paired = resident && ck.paired && segments_paired(w);
  auto length = [&](int s) {
    return (s + 1 < ck.nseg ? every : pl.nt - s * every);
  };
  auto set = [&](int s) -> void* { return ck.seg(paired ? (s & 1) * every : 0); };
  auto recompute = [&](int s) {
    return SegRecompute{ck.a(s), ck.b(s), pl.s[3], ck.seg(ck.nvol - 1), set(s), length(s)};
  };
  if (paired) {
    const SegRecompute last = recompute(ck.nseg - 1);
    bool refused = false;
    rc = launch_segments(w, &last, nullptr, ck.vol / 4, st, &refused);
    if (rc != FFPAT_OK && !refused) return rc;
    if (refused) resident = false;
  }
  for (int s = ck.nseg - 1; s >= 0; --s) {
    const int lo = s * every;
    const int hi = (lo + every - 1 < pl.nt - 1) ? lo + every - 1 : pl.nt - 1;
    if (resident) {
      const int steps = length(s);
      int x, y;
      others(&x, &y);
      const SegTranspose tr{B[u], B[v], B[x], B[y], ck.acc(), set(s), steps, lo == 0};
      bool refused = false;
      if (paired) {
        const SegRecompute before = s > 0 ? recompute(s - 1) : SegRecompute{};
        rc = launch_segments(w, s > 0 ? &before : nullptr, &tr, ck.vol / 4, st, &refused);
      } else {
        const SegRecompute now = recompute(s);
        rc = launch_segments(w, &now, nullptr, ck.vol / 4, st, &refused);
        if (rc == FFPAT_OK) rc = launch_segments(w, nullptr, &tr, ck.vol / 4, st, &refused);
      }
      if (rc != FFPAT_OK && !refused) return rc;
      resident = !refused;  // refused: this segment and the rest launch by launch
    }
    if (resident) {
      const int steps = length(s);
      int x, y;
      others(&x, &y);
      const int last = (steps - 1) & 1 ? y : x, prev = (steps - 1) & 1 ? x : y;
      v = steps > 1 ? prev : u;  // mu^{lo+1}
      u = last;                  // mu^{lo}
      if (lo == 0) end = B[u];
      continue;
    }
    auto P = [&](int j) -> void* { return j == 0 ? ck.a(s) : (j == 1 ? ck.b(s) : ck.seg(j)); };
    // recompute p^{lo+2} .. p^{hi} from the checkpoint, two steps per pass
    // where allowed
    for (int j = 1; j + 1 <= hi - lo;) {
      if (two && j + 2 <= hi - lo) {
        rc = launch_step2_f32(w, P(j - 1), P(j), P(j + 1), P(j + 2), st);
        j += 2;
      } else {
        rc = step3(w, tma, false, P(j), P(j - 1), P(j + 1), nullptr, st);
        j += 1;
      }
      if (rc != FFPAT_OK) return rc;
    }
    for (int n = hi; n >= lo;) {
      const void* pn = P(n - lo);
      if (two_t && n - 1 >= lo && n - 1 >= 1) {
        // mu^n, mu^{n-1} in one pass; the accumulations in the order of
        // the single steps (mu^{n+1} L(p^n), then mu^n L(p^{n-1}))
        int x, y;
        others(&x, &y);
        rc = launch_step2_f32(w, B[v], B[u], B[x], B[y], st);
        if (rc == FFPAT_OK) rc = launch_lap_accum(w, ck.acc(), B[u], pn, 1.0, st);
        if (rc == FFPAT_OK) rc = launch_lap_accum(w, ck.acc(), B[x], P(n - 1 - lo), 1.0, st);
        if (rc != FFPAT_OK) return rc;
        u = y;  // mu^{n-1}
        v = x;  // mu^n
        n -= 2;
      } else if (n >= 1) {
        rc = launch_lap_accum(w, ck.acc(), B[u], pn, 1.0, st);
        if (rc == FFPAT_OK) rc = step3(w, tma, false, B[u], B[v], B[v], nullptr, st);  // mu^n
        if (rc != FFPAT_OK) return rc;
        const int t = u;
        u = v;
        v = t;
        n -= 1;
      } else {
        rc = launch_lap_accum(w, ck.acc(), B[u], pn, 0.5, st);
        if (rc == FFPAT_OK) rc = step3(w, tma, true, B[u], nullptr, ck.seg(0), nullptr, st);
        if (rc != FFPAT_OK) return rc;
        tmp = ck.seg(0);
        n -= 1;
      }
    }
  }
  // grad_h = (start(mu^1) - mu^2) / (kappa / 12), grad_c = 2 acc / c, on dense rows
  if (grad_h)
    rc = end ? launch_kscale(pl, end, grad_h, false, st)
             : launch_sub_div(pl, tmp, B[v], grad_h, st);
  if (rc != FFPAT_OK || !grad_c) return rc;
  return launch_scale_div(pl, ck.acc(), c, 2.0, grad_c, st);
}

}  // extern "C"
