// Host-side tensor-contraction engine: device buffers, workspace, einsum-style
// contractions mapped onto the strided complex GEMM, permutes and vector helpers.
#pragma once
#include <functional>
#include <memory>
#include <string>
#include <vector>

#include "f64_tc.cuh"
#include "kernels.cuh"

namespace cclr {

// Device memory charged to one owner (a context): bytes held now, the most ever held, and
// an optional limit (0 = none) that every allocation charged to it is checked against.
struct MemAcct {
  size_t used = 0, peak = 0, budget = 0;
  // frees what the owner keeps only for speed; true if anything was freed.  An allocation that fails or
  // would exceed the budget calls it and tries once more.
  std::function<bool()> reclaim;
};
// The account that allocations made on this thread are charged to (nullptr: none).
MemAcct *&current_acct();
// Charges the allocations of a scope (one library call) to an account.
struct AcctScope {
  MemAcct *prev;
  explicit AcctScope(MemAcct *a) : prev(current_acct()) { current_acct() = a; }
  ~AcctScope() { current_acct() = prev; }
  AcctScope(const AcctScope &) = delete;
  AcctScope &operator=(const AcctScope &) = delete;
};

// Owning device allocation.  An allocation over the current account's budget (after its reclaim) throws
// status 2 (CCLR_ENOMEM) before cudaMalloc is called; the bytes are returned to the same account when
// the buffer is released, whichever thread releases it.
struct DevBuf {
  void *p = nullptr;
  size_t bytes = 0;
  MemAcct *acct = nullptr;
  DevBuf() = default;
  explicit DevBuf(size_t b) { alloc(b); }
  DevBuf(const DevBuf &) = delete;
  DevBuf &operator=(const DevBuf &) = delete;
  DevBuf(DevBuf &&o) noexcept : p(o.p), bytes(o.bytes), acct(o.acct) { o.p = nullptr; o.bytes = 0; o.acct = nullptr; }
  DevBuf &operator=(DevBuf &&o) noexcept {
    if (this != &o) {
      release();
      p = o.p; bytes = o.bytes; acct = o.acct;
      o.p = nullptr; o.bytes = 0; o.acct = nullptr;
    }
    return *this;
  }
  ~DevBuf() { release(); }
  void alloc(size_t b);
  void release();
  template <typename T> T *as() const { return (T *)p; }
};

// The tiles of a ladder group's formation W[(b, f)][(a, e)] (b and a counted from the group's first a, v rows and
// columns each) that hold an entry with b > a, which are all that is read of it: a group of g values of a computes
// g (g + 1) / 2 of the v g blocks less (a fifth of the work at v = 160, g = 32).  Lists are made once per tiling and
// kept; get() returns nullptr (compute every tile) where it cannot make one (no memory, inside a capture).
class UpperTiles {
 public:
  explicit UpperTiles(int v = 1) : v_(v) {}
  // nMt x nNt tiles of rows x cols entries from row m0 and column n0 on, of M rows in all, in bands of `band` tile
  // rows; *n: tiles in the list
  const uint32_t *get(int nMt, int nNt, int band, int rows, int cols, int64_t m0, int64_t n0, int64_t M, cudaStream_t st,
                      int *n);
  void reset(int v) {
    lists_.clear();
    v_ = v;
  }

 private:
  struct List {
    int nMt, nNt, band, rows, cols, n;
    int64_t m0, n0, M;
    DevBuf buf;
  };
  std::vector<std::unique_ptr<List>> lists_;
  int v_;
};

size_t device_bytes_in_use();
// Counter bumped whenever device memory is freed (and by callers that rewrite state a captured
// CUDA graph depends on): a graph captured at one value is valid while the counter keeps it.
unsigned long long state_epoch();
void bump_state_epoch();

class Engine {
 public:
  cudaStream_t st = nullptr;
  // complex64 contractions above a size threshold run on the tcgen05 tensor cores:
  // 0 = never (CUDA-core FP32), 1 = TF32, 2 = 3xTF32 split, 3 = bf16x3 split.
  int tc_mode = 0;
  bool tc_force = false;  // route every complex64 contraction to the tensor cores (self-test)
  int64_t tc_calls = 0;
  // Workspace slot s of at least `bytes` bytes (grown on demand, reused across calls).
  void *ws(int slot, size_t bytes);
  // frees the workspace slots (they grow again on demand)
  void release_ws() {
    slots_.clear();
    f64_slots_.clear();
    f64_scr_.release();
  }
  // C[mc] += alpha * sum A[ma] B[mb] over the modes not in mc (einsum semantics; every
  // mode must appear in exactly two operands or in all three).
  void contract(zc alpha, const Tens &A, const std::string &ma, const Tens &B,
                const std::string &mb, const Tens &C, const std::string &mc);
  // the complex64 tensor-core branch of contract (modes already classified)
  void contract_tc(zc alpha, const Tens &A, const std::string &ma, const Tens &B, const std::string &mb,
                   const Tens &C, const std::string &mc, const std::string &bat, const std::string &Mm,
                   const std::string &Nm, const std::string &Km, int64_t nb, int64_t M, int64_t N, int64_t K);
  // the complex128 tensor-core branch (f64_tc.cuh); false: no memory for the operands' slices, nothing done
  bool contract_f64(zc alpha, const Tens &A, const std::string &ma, const Tens &B, const std::string &mb, const Tens &C,
                    const std::string &mc, const std::string &bat, const std::string &Mm, const std::string &Nm,
                    const std::string &Km, int64_t nb, int64_t M, int64_t N, int64_t K);
  // Slices of a complex128 operand (f64tc_prep) in workspace slot `slot`, or, with a key, kept until
  // clear_prep_cache() like the other constant operands (at most f64_cache_cap bytes).  Throws status 2.
  F64Op f64_operand(int slot, const void *src, View2 rv, View2 kv, int64_t R, int64_t K, bool embed,
                    const std::string &key);
  // the kept slices of an operand (made here if there is room to keep them); false, and nothing done, where there is none
  bool f64_kept(const void *src, View2 rv, View2 kv, int64_t R, int64_t K, bool embed, const std::string &key, F64Op &op);
  // room for the sums of f64tc_gemms of up to M x N (throws status 2), and a product itself on this engine's stream; the
  // room has to be claimed before: nothing is allocated, and so nothing can fail, between the products of a call
  void f64_scratch(int64_t M, int64_t N);
  void f64_gemm(const F64Op &A, int64_t M, const F64Op &B, int64_t N, int64_t K, void *C, View2 rv, View2 cv, zc alpha,
                bool accumulate, UpperTiles *upper = nullptr, int64_t upper_row = 0, int64_t upper_col = 0);
  // Throws status 5 if a tensor-core kernel launched since the last check gave up on a bounded wait
  // (synchronises the stream; nothing is done when none was launched).
  void check_tc();
  bool tc_pending = false;
  // claims workspace slot `slot` for R rows of K entries.  Throws status 2.
  void f64_reserve(int slot, int64_t R, int64_t K, bool embed);
  size_t f64_cache_cap = 0;
  int64_t f64_operand_cap = 2ll << 30;  // bytes of an operand's slices that are not kept: in chunks above that
  // Holds off f64_reclaim() while prepared slices are in use on the host side.
  struct F64Hold {
    Engine &e;
    explicit F64Hold(Engine &e_) : e(e_) { ++e.f64_holds_; }
    ~F64Hold() { --e.f64_holds_; }
    F64Hold(const F64Hold &) = delete;
  };
  // frees the FP64 slices (workspace and kept operands); true if there were any
  bool f64_reclaim();
  // out[mo] (+)= alpha * in[mi]  (same mode set; dtypes may differ -> conversion).
  void permute(zc alpha, const Tens &in, const std::string &mi, const Tens &out,
               const std::string &mo, bool acc);
  void zero(const Tens &t);
  double2 *dot_scratch();  // device: partials [>=304] and results [64]
  double2 *dot_results();
  // Constant operands: while cst_hint points at one operand of a tensor-core contraction, the
  // prepared form of that operand (its permuted copy, its TF32 / BF16 embedded rows or columns, or its
  // FP64 slices) is kept and reused by later contractions of the same operand with the same modes and
  // precision; at most prep_cache_cap (f64_cache_cap) bytes (0: off).  Whoever rewrites or frees a
  // constant calls clear_prep_cache() before and after.
  const void *cst_hint = nullptr;
  size_t prep_cache_cap = 0;
  void clear_prep_cache() {
    prep_.clear();
    prep_bytes_ = 0;
    f64_kept_.clear();
    f64_kept_bytes_ = 0;
  }
  size_t prep_cache_bytes() const { return prep_bytes_; }

 private:
  std::vector<DevBuf> slots_;
  DevBuf dots_;
  struct PrepEntry {
    std::string key;
    DevBuf buf;
    bool filled = false;
  };
  std::vector<std::unique_ptr<PrepEntry>> prep_;
  size_t prep_bytes_ = 0;
  // a valid entry, or nullptr
  PrepEntry *prep_find(const std::string &key);
  // the entry to (re)fill, created if needed; nullptr when it would exceed the cap
  PrepEntry *prep_get(const std::string &key, size_t bytes);
  // the kept entry of that key and size, created if needed; nullptr where there is no room to keep it
  PrepEntry *f64_keep(const std::string &key, size_t bytes);
  std::vector<DevBuf> f64_slots_;  // slices, then tops in the same buffer
  std::vector<std::unique_ptr<PrepEntry>> f64_kept_;  // slices, then tops in the same buffer
  size_t f64_kept_bytes_ = 0;
  DevBuf f64_scr_;
  F64Side f64_side_;
  int f64_holds_ = 0;
};

}  // namespace cclr
