// Host run of the transforms on pairs of components (fft_pair.cuh): RegPlan::run on pairs and on strided
// lines, RegPlan::run_regrouped (threads change places at one exchange), Fft16 and the inverse row transform of
// FFT length 768 (s3_rows_inverse), for the CPU test suite.
//
// The lanes are cooperative fibers of one host thread. A fiber runs until a barrier stops it, and the scheduler
// always takes the first fiber that can run, in ascending or in descending order. So between two barriers
// every lane does all of its shared-memory accesses before or after those of any other lane, whichever is the
// worse: an access that no barrier separates from another lane's write of the same place gives a
// wrong result in one of the two orders, every time. A lane waits only for the lanes of its own line (the GPU's
// warp barrier may wait for more), or for all of the group where the kernels meet at a CTA barrier.
//
// Usage: fft_pair_host <out.bin>. A record per line and component: eight int32 values (kind, L, V, INV,
// HIN, order, inputs, outputs), then the input and the output as complex128. Kinds: 0 run, 1 run on a strided
// line, 2 run_regrouped at exchange 0, 3 at the last exchange, 4 Fft16, 5 length-768 rows.
#include <ucontext.h>

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <functional>
#include <map>
#include <vector>

#include "../../paper_2402_02116_gb300/csrc/fft16.cuh"
#include "../../paper_2402_02116_gb300/csrc/op_split3.cuh"

using namespace dbi;

namespace {

class Fibers {
 public:
  struct Barrier {  // over `size` lanes of group `id`
    Fibers *f;
    int id, size;
    void operator()() const { f->wait(id, size); }
  };
  Barrier barrier(int id, int size) { return {this, id, size}; }

  // body(lane) for every lane; false if lanes are left waiting at a barrier.
  bool run(int n, bool descending, std::function<void(int)> body) {
    lanes_.assign(n, Lane{});
    groups_.clear();
    body_ = std::move(body);
    self() = this;
    for (int i = 0; i < n; ++i) {
      Lane &l = lanes_[i];
      l.stack.resize(kStack);
      getcontext(&l.ctx);
      l.ctx.uc_stack.ss_sp = l.stack.data();
      l.ctx.uc_stack.ss_size = kStack;
      l.ctx.uc_link = &main_;
      makecontext(&l.ctx, reinterpret_cast<void (*)()>(&Fibers::entry), 1, i);
    }
    for (;;) {
      int next = -1;
      for (int k = 0; k < n && next < 0; ++k) {
        const int i = descending ? n - 1 - k : k;
        const Lane &l = lanes_[i];
        if (!l.done && (l.group < 0 || groups_[l.group].generation != l.generation)) next = i;
      }
      if (next < 0) break;
      current_ = next;
      lanes_[next].group = -1;
      swapcontext(&main_, &lanes_[next].ctx);
    }
    for (const Lane &l : lanes_)
      if (!l.done) return false;
    return true;
  }

 private:
  static constexpr size_t kStack = 128 * 1024;
  struct Lane {
    ucontext_t ctx;
    std::vector<char> stack;
    bool done = false;
    int group = -1, generation = 0;  // the barrier it waits at
  };
  struct Group {
    int arrived = 0, generation = 0;
  };
  static Fibers *&self() {
    static Fibers *f = nullptr;
    return f;
  }
  static void entry(int i) {
    self()->body_(i);
    self()->lanes_[i].done = true;
  }
  void wait(int id, int size) {
    Group &g = groups_[id];
    if (++g.arrived == size) {
      g.arrived = 0;
      ++g.generation;
      return;
    }
    Lane &l = lanes_[current_];
    l.group = id;
    l.generation = g.generation;
    swapcontext(&l.ctx, &main_);
  }
  std::vector<Lane> lanes_;
  std::map<int, Group> groups_;
  std::function<void(int)> body_;
  ucontext_t main_;
  int current_ = 0;
};

FILE *g_out;
std::vector<float2> g_tw;
uint64_t g_seed = 1;
bool g_ok = true;

float uniform() {
  g_seed = g_seed * 6364136223846793005ULL + 1442695040888963407ULL;
  return float(double(g_seed >> 11) / double(1ULL << 53) * 2.0 - 1.0);
}

using Line = std::vector<cpair>;
Line random_line(int n, int nonzero) {
  Line x(n, pzero());
  for (int i = 0; i < nonzero; ++i) {
    const float2 a = make_float2(uniform(), uniform()), b = make_float2(uniform(), uniform());
    x[i] = mkpair(a, b);
  }
  return x;
}

// Shared memory of a case, between guards that must stay untouched.
struct Memory {
  static constexpr int kGuard = 64;
  static constexpr pair64 kMark = 0x7123456789abcdefull;
  Line all;
  explicit Memory(size_t n) : all(n + 2 * kGuard, cpair{kMark, kMark}) {}
  cpair *data() { return all.data() + kGuard; }
  void check(const char *what, int L) const {
    for (int i = 0; i < kGuard; ++i)
      if (all[i].re != kMark || all[all.size() - 1 - i].re != kMark) {
        std::fprintf(stderr, "%s, L = %d: guard overwritten\n", what, L);
        g_ok = false;
      }
  }
};

void record(int kind, int L, int V, bool inv, bool hin, bool desc, const Line &in, const Line &out) {
  for (int c = 0; c < 2; ++c) {
    const int32_t h[8] = {kind, L, V, inv, hin, desc, int32_t(in.size()), int32_t(out.size())};
    std::fwrite(h, sizeof(h), 1, g_out);
    for (const Line *l : {&in, &out})
      for (const cpair &p : *l) {
        const float2 v = c ? comp1(p) : comp0(p);
        const double z[2] = {v.x, v.y};
        std::fwrite(z, sizeof(z), 1, g_out);
      }
  }
}
void must(bool ran, const char *what, int L) {
  if (ran) return;
  std::fprintf(stderr, "%s, L = %d: lanes left at a barrier\n", what, L);
  g_ok = false;
}

// One thread group transforming NLT lines (STRIDE > 1: elements STRIDE apart).
template <int L, int V, bool INV, bool HIN, int NLT, int STRIDE = 1> void plain(bool desc) {
  constexpr int T = L / 8, LP = RegFFT<cpair, L>::LP;
  std::vector<Line> in, out(NLT, Line(L));
  for (int l = 0; l < NLT; ++l) in.push_back(random_line(L, HIN ? L / 2 : L));
  Memory mem(size_t(NLT) * LP * STRIDE);
  Fibers fb;
  must(fb.run(T, desc, [&](int t) {
    const TwReg<float2, L, V> tr(t, g_tw.data());
    cpair v[NLT][8];
    for (int l = 0; l < NLT; ++l)
      for (int m = 0; m < 8; ++m) v[l][m] = in[l][t + m * T];
    const auto sync = fb.barrier(0, T);
    if constexpr (STRIDE == 1) {
      cpair *lines[NLT];
      for (int l = 0; l < NLT; ++l) lines[l] = mem.data() + size_t(l) * LP;
      RegPlan<L, V>::template run<cpair, NLT, INV, HIN>(v, lines, t, tr, sync);
    } else {
      const StridedLine<cpair> lines[1] = {{mem.data(), STRIDE}};
      RegPlan<L, V>::template run<cpair, 1, INV, HIN>(v, lines, t, tr, sync);
    }
    for (int l = 0; l < NLT; ++l)
      for (int m = 0; m < 8; ++m) out[l][t + m * T] = v[l][m];
  }), "run", L);
  mem.check("run", L);
  for (int l = 0; l < NLT; ++l) record(STRIDE > 1, L, V, INV, HIN, desc, in[l], out[l]);
}

// ROWS rows side by side, as the row stages: forward ones end, inverse ones begin with thread (row, t) =
// (i % ROWS, i / ROWS).
template <int L, int V, bool INV, bool HIN, int NLT> void regrouped(bool desc) {
  constexpr int T = L / 8, ROWS = 256 / T, PLP = row_pitch<L, ROWS>, X = INV ? 0 : PlanInfo<L, V>::np - 2;
  std::vector<Line> in, out(NLT * ROWS, Line(L));
  for (int l = 0; l < NLT * ROWS; ++l) in.push_back(random_line(L, HIN ? L / 2 : L));
  Memory mem(size_t(NLT) * ROWS * PLP);
  Fibers fb;
  must(fb.run(ROWS * T, desc, [&](int i) {
    const int rr = i / T, t = i % T, r = i % ROWS, tq = i / ROWS;  // the places along a row and across the rows
    const int ra = INV ? r : rr, ta = INV ? tq : t, rb = INV ? rr : r, tb = INV ? t : tq;
    const TwReg<float2, L, V> tr(INV ? t : ta, INV ? t : tb, g_tw.data());
    cpair v[NLT][8], *la[NLT], *lb[NLT];
    for (int l = 0; l < NLT; ++l) {
      la[l] = mem.data() + (size_t(l) * ROWS + ra) * PLP;
      lb[l] = mem.data() + (size_t(l) * ROWS + rb) * PLP;
      for (int m = 0; m < 8; ++m) v[l][m] = in[l * ROWS + ra][ta + m * T];
    }
    RegPlan<L, V>::template run_regrouped<cpair, NLT, INV, X, HIN>(v, la, ta, lb, tb, tr, fb.barrier(1 + rr, T),
                                                                   fb.barrier(0, ROWS * T));
    for (int l = 0; l < NLT; ++l)
      for (int m = 0; m < 8; ++m) out[l * ROWS + rb][tb + m * T] = v[l][m];
  }), "run_regrouped", L);
  mem.check("run_regrouped", L);
  for (int l = 0; l < NLT * ROWS; ++l) record(INV ? 2 : 3, L, V, INV, HIN, desc, in[l], out[l]);
}

template <int L, bool INV, bool HALF> void sixteen(bool desc) {
  using F = Fft16<L>;
  const Line in = random_line(L, HALF ? L / 2 : L);
  Line out(L);
  Memory mem(F::LP);
  Fibers fb;
  must(fb.run(F::T, desc, [&](int t) {
    const typename F::Base base(t, g_tw.data());
    cpair v[16];
    for (int m = 0; m < 16; ++m) v[m] = in[t + m * F::T];
    F::template run<INV, HALF>(v, mem.data(), t, base, fb.barrier(0, F::T));
    for (int m = 0; m < 16; ++m) out[t + m * F::T] = v[m];
  }), "Fft16", L);
  mem.check("Fft16", L);
  record(4, L, 0, INV, HALF, desc, in, out);
}

void rows768(bool desc) {
  std::vector<Line> in, out(kS3Units, Line(kS3L / 2));
  for (int r = 0; r < kS3Units; ++r) in.push_back(random_line(kS3L, kS3L));
  Memory mem(s3_smem() / sizeof(cpair));
  Fibers fb;
  must(fb.run(kS3Threads, desc, [&](int i) {
    const S3Place at = s3_place(i);
    const TwReg<float2, kS3M, 0> tr(i % kS3T, g_tw.data());
    cpair v[1][8], y[4];
    for (int m = 0; m < 8; ++m) v[0][m] = in[at.r][3 * (at.tq + m * kS3T) + at.qs];
    s3_rows_inverse(v, mem.data(), i, tr, g_tw.data(), y, fb.barrier(1 + i / kS3T, kS3T), fb.barrier(0, kS3Threads));
    for (int k = 0; k < 4; ++k) out[i / kS3UnitThreads][i % kS3UnitThreads + k * kS3UnitThreads] = y[k];
  }), "length-768 rows", kS3L);
  mem.check("length-768 rows", kS3L);
  for (int r = 0; r < kS3Units; ++r) record(5, kS3L, 0, true, false, desc, in[r], out[r]);
}

template <int L, int V> void length(bool desc) {
  plain<L, V, false, true, 1>(desc);
  plain<L, V, true, false, 1>(desc);
  plain<L, V, false, false, 2>(desc);
  regrouped<L, V, false, true, 1>(desc);
  regrouped<L, V, true, false, 1>(desc);
}

}  // namespace

int main(int argc, char **argv) {
  if (argc != 2 || !(g_out = std::fopen(argv[1], "wb"))) return 2;
  for (int m = 0; m < kTwiddleN; ++m) {
    const double a = -2.0 * M_PI * double(m) / double(kTwiddleN);
    g_tw.push_back(make_float2(float(std::cos(a)), float(std::sin(a))));
  }
  for (const bool desc : {false, true}) {
    length<16, 0>(desc);
    length<16, 1>(desc);
    length<32, 0>(desc);
    length<32, 1>(desc);
    length<64, 0>(desc);
    length<128, 0>(desc);
    length<128, 1>(desc);
    length<256, 0>(desc);
    length<256, 1>(desc);
    length<512, 0>(desc);
    regrouped<512, 0, false, false, 2>(desc);  // length 1024: both parities of a row
    regrouped<512, 0, true, false, 2>(desc);
    plain<16, 0, false, true, 1, 20>(desc);  // the z lines of the 3D slab: elements a row apart
    plain<32, 0, true, false, 1, 36>(desc);
    plain<64, 0, false, true, 1, 68>(desc);
    plain<128, 0, true, false, 1, 20>(desc);
    sixteen<32, false, true>(desc);
    sixteen<32, true, false>(desc);
    sixteen<64, false, true>(desc);
    sixteen<64, true, false>(desc);
    sixteen<128, false, true>(desc);
    sixteen<128, true, false>(desc);
    sixteen<256, false, true>(desc);
    sixteen<256, true, false>(desc);
    rows768(desc);
  }
  std::fclose(g_out);
  return g_ok ? 0 : 1;
}
