// Host task scheduler: turns the recursive H-LU of Algorithm 1 step II (block
// form: LU(A11); A12 <- L11^-1 P A12; A21 <- A21 U11^-1; A22 <- A22 - A21 A12
// truncated; LU(A22), as in the H-LU source the paper cites) and the
// preconditioner application U^-1 (L^-1 r) of step III into task DAGs.
//
// The recursion is walked once on the host.  Every leaf-level operation becomes
// a task of one of the kinds in hlu_internal.h; the data it touches is
// recorded per (buffer, leaf-cluster segment), which yields read-after-write,
// write-after-read and write-after-write edges.  The emission order is the
// sequential program order, hence a topological order: the device executor
// hands out tasks in that order and each task only waits on earlier ones.
//
// Ranks of low-rank blocks are data dependent.  The schedule only uses rank
// capacities; kernels read the live rank from a rank slot when they run.
#include <sys/mman.h>

#include <algorithm>
#include <chrono>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <future>
#include <queue>
#include <stdexcept>
#include <unordered_map>
#include <utility>

#include "hlu_internal.h"

namespace hlu {
namespace {

// The schedule's vectors reach gigabytes (n = 24: 2.2 GB of tasks, 1.2 GB of
// terms, 0.9 GB of predecessor indices), and every reallocation writes its
// new block once.  Growing by 4 instead of 2 writes about 4/3 of the final
// size instead of about 2x, which took a quarter off the n = 24 build (most
// of it page faults); the unused capacity is address space only.  Blocks of
// some megabytes ask for huge pages where the system gives them on request.
template <class V>
inline void grow4(V& v, size_t extra = 1) {
  if (v.size() + extra <= v.capacity()) return;
  v.reserve(std::max<size_t>(v.size() + extra, std::max<size_t>(4096, v.capacity() * 4)));
#ifdef MADV_HUGEPAGE
  constexpr uintptr_t kHuge = uintptr_t(1) << 21;
  const uintptr_t lo = ((uintptr_t)(v.data() + v.size()) + kHuge - 1) & ~(kHuge - 1);
  const uintptr_t hi = (uintptr_t)(v.data() + v.capacity()) & ~(kHuge - 1);
  if (hi > lo) madvise((void*)lo, hi - lo, MADV_HUGEPAGE);
#endif
}

constexpr int64_t kNotTemp = INT64_MAX;
struct MV {
  int32_t buf;   // dependency buffer (-1: read-only, untracked)
  int32_t clus;  // cluster whose index range the rows cover
  View v;
  int64_t at = kNotTemp;  // a temporary's position in the ring, counted over its passes
};
struct LR {
  MV X, Y;
};
struct PieceMV {
  LR p;
  int32_t xoff, yoff;
  float sign;
  int32_t win0 = 0, nwin = 0;  // a dense sum: the dependency buffers of its windows
};

// A dependency buffer: its segments, the tasks that touched it, and of a
// temporary the fences of its memory and where that lies in the ring.
struct Buf {
  int32_t base_leaf;
  int32_t nseg;
  int64_t seg0;
  int64_t acc_head = -1;   // list of accesses (acc_task_, acc_next_)
  int64_t fence_begin = 0;  // fences in fence_pool_
  int32_t n_fences = 0;
  int32_t acc_last = -1;    // the last task on the list
  int32_t chunk = -1, pass = 0;  // a temporary's first chunk (else -1) and its pass
};
struct Seg {
  int32_t writer = -1;
  int32_t buf = -1;
  int64_t rhead = -1;  // readers since (rtask_, rnext_)
};

// Pieces per truncation of accumulated updates (beside the target itself).
// Larger batches truncate less often; smaller ones leave less work to the task
// that the newest piece completes (n = 24 factorisation: 4 pieces 881 ms, 8
// pieces 709 ms, 16 pieces 782 ms).
constexpr size_t kBatch = 8;
constexpr size_t kDirect = 4;  // more pieces of a small target are summed densely first
constexpr size_t kDenseBatch = 16;  // pieces per dense update

// Targets of a subdivided x subdivided product up to this size on both sides
// are agglomerated in one truncation (the executor's dense route handles them
// whole); larger ones quadrant by quadrant first.
constexpr int32_t kOneStepAgglomeration = 128;

// A ring too small for the temporaries that a schedule holds.
struct RingFull : std::runtime_error {
  RingFull() : std::runtime_error("temporaries of one block's update exceed the ring") {}
};

class Sched {
 public:
  // accumulate: see gemm
  Sched(const std::vector<Cluster>& C, const std::vector<Block>& B, int32_t kcap, ArenaLayout& L,
        Schedule* S, std::vector<int32_t>& dbuf, std::vector<int32_t>& xbuf,
        std::vector<int32_t>& ybuf, bool make_buffers, int32_t segsz, bool accumulate,
        int64_t ring_off, int64_t ring_size)
      : C_(C), B_(B), kcap_(kcap), L_(L), S_(S), dbuf_(dbuf), xbuf_(xbuf), ybuf_(ybuf),
        ring_off_(ring_off), ring_size_(ring_size), accumulate_(accumulate) {
    S_->pred_ptr.assign(1, 0);
    updates_.resize(B_.size());
    // dependency segments: clusters of at most `segsz` DOFs whose parent is
    // larger (the tile level, or the leaves); every cluster covers a range of them
    seg_begin_.assign(C_.size(), 0);
    seg_end_.assign(C_.size(), 0);
    seg_cluster_.clear();
    segsz_ = segsz;
    assign_segments(0, false, segsz);
    for (chunk_ = 1 << 14; chunk_ < (1 << 18) && chunk_ * 8192 < ring_size_;) chunk_ *= 2;
    chunk_occ_.assign((size_t)((ring_size_ + chunk_ - 1) / chunk_) + 1, std::vector<int32_t>());
    chunk_fence_task_.assign(chunk_occ_.size(), -1);
    chunk_pass_.assign(chunk_occ_.size(), 0);
    if (make_buffers) {
      dbuf_.assign(B_.size(), -1);
      xbuf_.assign(B_.size(), -1);
      ybuf_.assign(B_.size(), -1);
    }
    // each schedule tracks its own buffer states from scratch
    for (size_t b = 0; b < B_.size(); ++b) {
      if (B_[b].kind == KIND_DENSE) dbuf_[b] = new_buf_single();
      if (B_[b].kind == KIND_ADM) {
        xbuf_[b] = new_buf_leaves(B_[b].row);
        ybuf_[b] = new_buf_leaves(B_[b].col);
      }
    }
  }

  // ---------------------------------------------------------------- segments
  void assign_segments(int32_t c, bool inside, int32_t segsz) {
    const Cluster& cl = C_[c];
    bool is_seg = !inside && (cl.size <= segsz || cl.son[0] < 0);
    if (is_seg || inside) {
      if (is_seg) seg_cluster_.push_back(c);
      int32_t sidx = (int32_t)seg_cluster_.size() - 1;
      seg_begin_[c] = sidx;
      seg_end_[c] = sidx + 1;
      if (cl.son[0] >= 0) {
        assign_segments(cl.son[0], true, segsz);
        assign_segments(cl.son[1], true, segsz);
      }
      return;
    }
    seg_begin_[c] = (int32_t)seg_cluster_.size();
    assign_segments(cl.son[0], false, segsz);
    assign_segments(cl.son[1], false, segsz);
    seg_end_[c] = (int32_t)seg_cluster_.size();
  }

  // ---------------------------------------------------------------- arena
  // Temporaries live in a ring region.  Re-using ring memory orders the new
  // occupant's writers after every task that touched the memory before.
  // A fence orders one chunk of the ring: 1/8192 of it, between 2^14 and 2^18
  // elements (n = 24, 10 passes over 2^31: 1.29 M fences in chunks of 2^14, 80
  // thousand in chunks of 2^18).
  int64_t chunk_ = 0;
  int64_t alloc(int64_t n) {
    n = (n + 31) & ~int64_t(31);
    temp_elems_ += n;
    if (n > ring_size_) throw RingFull();
    add_old_pieces(n);
    if (cursor_ + n > ring_size_) {
      cursor_ = 0;
      ++pass_;
      ++wraps_;
    }
    int64_t o = cursor_;
    last_alloc_pos_ = ring_pos();
    cursor_ += n;
    pending_fence_.clear();
    for (int64_t ch = o / chunk_; ch <= (o + n - 1) / chunk_; ++ch) {
      if (chunk_pass_[ch] != pass_) {
        // first use of this chunk in this pass: a no-work fence task waits for
        // every task that touched the chunk's previous occupants
        chunk_fence_task_[ch] = -1;
        if (!chunk_occ_[ch].empty()) {
          Task f = make(TK_FENCE);
          int32_t saved_cur = cur_;
          std::vector<int32_t> saved_deps;
          saved_deps.swap(deps_);
          begin(f);
          for (int32_t old : chunk_occ_[ch])
            for (int64_t r = bufs_[old].acc_head; r >= 0; r = acc_next_[r]) dep(acc_task_[r]);
          end();
          chunk_fence_task_[ch] = cur_;
          deps_.swap(saved_deps);
          cur_ = saved_cur;
        }
        chunk_occ_[ch].clear();
        chunk_pass_[ch] = pass_;
      }
      if (chunk_fence_task_[ch] >= 0) pending_fence_.push_back(chunk_fence_task_[ch]);
    }
    last_alloc_lo_ = o / chunk_;
    last_alloc_hi_ = (o + n - 1) / chunk_;
    return ring_off_ + o;
  }
  // Positions in the ring count up over its passes.  A noted low-rank update
  // (settle) may hold factors in the ring for long: before the cursor comes
  // within a quarter of the ring of their memory, they are added to their
  // leaves (ready or not, the tasks wait for what they read).  The factors'
  // positions are kept in kBuckets buckets per pass.
  static constexpr int64_t kBuckets = 64;
  int64_t ring_pos() const { return pass_ * ring_size_ + cursor_; }
  static int64_t position(const LR& p) { return std::min(p.X.at, p.Y.at); }
  void add_old_pieces(int64_t n) {
    const int64_t bucket = (ring_size_ + kBuckets - 1) / kBuckets;
    const int64_t until = (ring_pos() + n - ring_size_ + ring_size_ / 4) / bucket;
    for (; forced_bucket_ <= until; ++forced_bucket_) {
      auto it = held_.find(forced_bucket_);
      if (it == held_.end()) continue;
      const std::vector<int32_t> blocks = std::move(it->second);
      held_.erase(it);
      for (int32_t c : blocks) {
        std::vector<Update> keep, old;
        for (Update& u : updates_[c])
          (u.a < 0 && position(u.p) / bucket <= forced_bucket_ ? old : keep).push_back(u);
        updates_[c].swap(keep);
        std::sort(old.begin(), old.end(), [](const Update& x, const Update& y) { return x.seq < y.seq; });
        std::vector<PieceMV> ps;
        for (const Update& u : old) ps.push_back(PieceMV{u.p, 0, 0, u.sign});
        early_pieces_ += (int64_t)ps.size();
        if (!ps.empty()) add_down(c, ps);
      }
    }
  }
  void add_down(int32_t c, const std::vector<PieceMV>& ps) {
    if (kind(c) != KIND_SUB) {
      add_pieces(c, ps, false);  // called while memory is being allocated
      return;
    }
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < 2; ++j) {
        std::vector<PieceMV> sp;
        for (const PieceMV& p : ps)
          sp.push_back(PieceMV{LR{sub(p.p.X, C_[rowc(c)].son[i]), sub(p.p.Y, C_[colc(c)].son[j])}, 0, 0, p.sign});
        add_down(son(c, i, j), sp);
      }
  }
  // a product a b (a >= 0) or a low-rank update p noted at a block
  struct Update {
    int32_t a = -1, b = -1;
    LR p;
    float sign = 0;
    int64_t seq = 0;  // when it arose: older updates are added first
  };
  void note_update(int32_t c, Update u, int64_t seq = -1) {
    u.seq = seq >= 0 ? seq : ++update_seq_;
    updates_[c].push_back(u);
    if (u.a >= 0) return;
    const int64_t at = position(u.p);
    if (at == kNotTemp) return;
    std::vector<int32_t>& h = held_[std::max(at / ((ring_size_ + kBuckets - 1) / kBuckets), forced_bucket_)];
    if (h.empty() || h.back() != c) h.push_back(c);
  }

  // attach the fence of the last allocation to buffer `b` and record it as
  // the occupant of that ring range
  void bind_alloc(int32_t b) {
    if (!pending_fence_.empty()) {
      std::sort(pending_fence_.begin(), pending_fence_.end());
      pending_fence_.erase(std::unique(pending_fence_.begin(), pending_fence_.end()), pending_fence_.end());
      bufs_[b].fence_begin = (int64_t)fence_pool_.size();
      bufs_[b].n_fences = (int32_t)pending_fence_.size();
      fence_pool_.insert(fence_pool_.end(), pending_fence_.begin(), pending_fence_.end());
      pending_fence_.clear();
    }
    for (int64_t ch = last_alloc_lo_; ch <= last_alloc_hi_; ++ch) chunk_occ_[ch].push_back(b);
    bufs_[b].chunk = (int32_t)last_alloc_lo_;
    bufs_[b].pass = pass_;
  }
  int32_t new_slot() { return L_.n_slots++; }
  int64_t temp_elems_ = 0;
  int64_t peak_ = 0;

  // ---------------------------------------------------------------- buffers
  int32_t push_buf(int32_t base_leaf, int32_t nseg) {
    const int32_t id = (int32_t)bufs_.size();
    Buf b;
    b.base_leaf = base_leaf;
    b.nseg = nseg;
    b.seg0 = (int64_t)segs_.size();
    Seg g;
    g.buf = id;
    grow4(segs_, nseg);
    segs_.resize(segs_.size() + nseg, g);
    grow4(bufs_);
    bufs_.push_back(b);
    return id;
  }
  int32_t new_buf_leaves(int32_t clus) { return push_buf(seg_begin_[clus], seg_end_[clus] - seg_begin_[clus]); }
  int32_t new_buf_single() { return push_buf(-1, 1); }

  // ---------------------------------------------------------------- views
  int32_t rowc(int32_t b) const { return B_[b].row; }
  int32_t colc(int32_t b) const { return B_[b].col; }
  int32_t sz(int32_t c) const { return C_[c].size; }
  int32_t kind(int32_t b) const { return B_[b].kind; }
  int32_t son(int32_t b, int i, int j) const { return B_[b].son[2 * i + j]; }

  MV mvD(int32_t b) const {
    MV m;
    m.buf = dbuf_[b];
    m.clus = rowc(b);
    m.v = View{L_.dense_off[b], 1, sz(rowc(b)), sz(rowc(b)), sz(colc(b)), -1, 0};
    return m;
  }
  MV mvDT(int32_t b) const {
    MV m;
    m.buf = dbuf_[b];
    m.clus = colc(b);
    m.v = View{L_.dense_off[b], sz(rowc(b)), 1, sz(colc(b)), sz(rowc(b)), -1, 0};
    return m;
  }
  MV mvX(int32_t b) const {
    MV m;
    m.buf = xbuf_[b];
    m.clus = rowc(b);
    m.v = View{L_.x_off[b], 1, sz(rowc(b)), sz(rowc(b)), L_.cap[b], L_.slot[b], 0};
    return m;
  }
  MV mvY(int32_t b) const {
    MV m;
    m.buf = ybuf_[b];
    m.clus = colc(b);
    m.v = View{L_.y_off[b], 1, sz(colc(b)), sz(colc(b)), L_.cap[b], L_.slot[b], 0};
    return m;
  }
  MV mvIdent(int32_t clus) const {
    if (sz(clus) > L_.ident_n) throw std::logic_error("identity too small");
    MV m;
    m.buf = -1;
    m.clus = clus;
    m.v = View{L_.ident_off, 1, L_.ident_n, sz(clus), sz(clus), -1, 0};
    return m;
  }
  MV sub(const MV& m, int32_t s) const {
    int32_t d = C_[s].off - C_[m.clus].off;
    if (d < 0 || d + C_[s].size > C_[m.clus].size) throw std::logic_error("sub view outside");
    MV r = m;
    r.clus = s;
    r.v.off += (int64_t)d * m.v.rs;
    r.v.rows = C_[s].size;
    return r;
  }
  // fresh temporary with per-leaf dependency segments; column count via a slot
  MV new_temp(int32_t clus, int32_t cols_cap) {
    MV m;
    m.clus = clus;
    int32_t rows = sz(clus);
    int64_t off = alloc((int64_t)rows * std::max(cols_cap, 1));
    m.at = last_alloc_pos_;
    m.buf = new_buf_leaves(clus);
    bind_alloc(m.buf);
    m.v = View{off, 1, rows, rows, cols_cap, new_slot(), 0};
    return m;
  }
  MV new_dense_temp(int32_t clus, int32_t cols) {
    MV m;
    m.clus = clus;
    int32_t rows = sz(clus);
    int64_t off = alloc((int64_t)rows * cols);
    m.at = last_alloc_pos_;
    m.buf = new_buf_single();
    bind_alloc(m.buf);
    m.v = View{off, 1, rows, rows, cols, -1, 0};
    return m;
  }
  int32_t cols_cap(const View& v) const { return v.cols; }

  // ---------------------------------------------------------------- tasks
  int32_t begin(const Task& t) {
    int32_t id = (int32_t)S_->tasks.size();
    grow4(S_->tasks);
    grow4(stamp_);
    grow4(implied_);
    S_->tasks.push_back(t);
    stamp_.push_back(-1);
    implied_.push_back(-1);
    cur_ = id;
    deps_.clear();
    return id;
  }
  void dep(int32_t p) {
    if (p < 0 || p == cur_) return;
    if (stamp_[p] == cur_) return;
    stamp_[p] = cur_;
    deps_.push_back(p);
  }
  // A temporary may be used until its first chunk is entered in a later pass of
  // the ring: the fence made then orders the chunk's next occupants after the
  // accesses noted so far, and no later one.
  void note_access(int32_t id) {
    Buf& b = bufs_[id];
    if (b.acc_last == cur_) return;
    if (b.chunk >= 0 && chunk_pass_[b.chunk] != b.pass) throw RingFull();
    b.acc_last = cur_;
    grow4(acc_task_);
    grow4(acc_next_);
    acc_task_.push_back(cur_);
    acc_next_.push_back(b.acc_head);
    b.acc_head = (int64_t)acc_task_.size() - 1;
  }
  void touch(int64_t seg, bool w) {
    Seg& g = segs_[seg];
    const Buf& b = bufs_[g.buf];
    if (g.writer < 0)
      for (int64_t f = b.fence_begin; f < b.fence_begin + b.n_fences; ++f) dep(fence_pool_[f]);
    note_access(g.buf);
    dep(g.writer);
    if (w) {
      for (int64_t r = g.rhead; r >= 0; r = rnext_[r]) dep(rtask_[r]);
      g.rhead = -1;
      g.writer = cur_;
    } else {
      grow4(rtask_);
      grow4(rnext_);
      rtask_.push_back(cur_);
      rnext_.push_back(g.rhead);
      g.rhead = (int64_t)rtask_.size() - 1;
    }
  }
  void acc(const MV& m, bool w) {
    if (m.buf < 0) return;
    const Buf& b = bufs_[m.buf];
    if (b.nseg == 1 && b.base_leaf < 0) {
      touch(b.seg0, w);
      return;
    }
    for (int32_t l = seg_begin_[m.clus]; l < seg_end_[m.clus]; ++l) {
      int64_t s = b.seg0 + (l - b.base_leaf);
      touch(s, w);
    }
  }
  // read of one segment: enough to order the task after any writer of the
  // buffer's rank slot (rank writers write every segment).  The right-hand
  // side count of a solve or apply is a launch parameter that no task
  // writes, so a count taken from it orders nothing: without this, every
  // update of the backward solve waited for the first segment of its input,
  // which is solved last
  void acc_rank(const MV& m) {
    if (m.buf < 0 || m.v.slot < 0 || m.v.slot == L_.nrhs_slot) return;
    const Buf& b = bufs_[m.buf];
    touch(b.seg0, false);
  }
  // Predecessors that another one already waits for order nothing more: they
  // are dropped when one of the kReduce latest predecessors lists them.  Every
  // edge left costs its finishing task an atomic (n = 24: 94 M edges with all of
  // them, 82 M without).  Lists are ascending: only their end, from this task's
  // first predecessor on, can name one of its predecessors.
  void end() {
    std::sort(deps_.begin(), deps_.end());
    if (deps_.size() > 1) {
      constexpr size_t kReduce = 8;
      const int32_t first = deps_.front();
      bool any = false;
      for (size_t k = 0; k < std::min(kReduce, deps_.size() - 1); ++k) {
        const int32_t q = deps_[deps_.size() - 1 - k];
        if (implied_[q] == cur_) continue;
        for (int64_t e = S_->pred_ptr[q + 1] - 1; e >= S_->pred_ptr[q] && S_->pred_idx[e] >= first; --e) {
          implied_[S_->pred_idx[e]] = cur_;
          any = true;
        }
      }
      if (any)
        deps_.erase(std::remove_if(deps_.begin(), deps_.end(), [&](int32_t p) { return implied_[p] == cur_; }),
                    deps_.end());
    }
    grow4(S_->pred_idx, deps_.size());
    grow4(S_->pred_ptr);
    S_->pred_idx.insert(S_->pred_idx.end(), deps_.begin(), deps_.end());
    S_->pred_ptr.push_back((int64_t)S_->pred_idx.size());
  }

  static Task make(int32_t type) {
    Task t;
    std::memset(&t, 0, sizeof(t));
    t.type = type;
    t.out_slot = -1;
    t.piv_off = -1;
    t.sign = 1.0f;
    t.a.slot = t.b.slot = t.c.slot = -1;
    return t;
  }

  // ---------------------------------------------------------------- leaf ops
  void getrf(int32_t d) {
    Task t = make(TK_GETRF);
    t.a = mvD(d).v;
    t.piv_off = L_.piv_off[d];
    begin(t);
    acc(mvD(d), true);
    end();
  }
  void trsm_leaf(int32_t type, int32_t d, const MV& V) {
    Task t = make(type);
    t.a = mvD(d).v;
    t.b = V.v;
    t.piv_off = L_.piv_off[d];
    begin(t);
    acc(mvD(d), false);
    acc(V, true);
    end();
  }

  // ---------------------------------------------------------------- H x multivector
  void leaves_of(int32_t b, std::vector<int32_t>& out) const {
    if (kind(b) != KIND_SUB) {
      out.push_back(b);
      return;
    }
    for (int k = 0; k < 4; ++k) leaves_of(B_[b].son[k], out);
  }

  // Vout (+)= sign * op(b) Vin, op = transpose when trans.  Vin covers the
  // in-cluster of b, Vout its out-cluster.  overwrite: Vout starts from zero
  // and out_slot receives Vin's column count.
  // late_seg >= 0 (accumulating): the terms of every output unit are split
  // into ROWMV tasks by how long before late_seg, the input's last segment
  // to be solved, their input is final: group 0 reads late_seg itself, group
  // g >= 1 segments 2^(g-1) to 2^g - 1 before it.  Far groups run first, so
  // only the few terms reading late_seg wait for the end of the preceding solve.
  void hmul(int32_t b, const MV& Vin, const MV& Vout, float sign, bool trans, bool overwrite, int32_t out_slot,
            int32_t late_seg = -1) {
    // (scratch of this call, kept for its capacity)
    std::vector<int32_t>&lv = hm_.leaves, &units = hm_.units, &cnt = hm_.cnt, &fill = hm_.fill, &items = hm_.items,
        &part = hm_.part;
    std::vector<MV>& T = hm_.T;
    std::vector<int8_t>& group = hm_.group;
    lv.clear();
    leaves_of(b, lv);
    int32_t oc = trans ? colc(b) : rowc(b);
    if (Vout.clus != oc || Vin.clus != (trans ? rowc(b) : colc(b)))
      throw std::logic_error("hmul cluster mismatch");
    T.resize(lv.size());
    for (size_t i = 0; i < lv.size(); ++i) {
      int32_t be = lv[i];
      if (kind(be) != KIND_ADM) continue;
      MV A = trans ? mvX(be) : mvY(be);
      int32_t ic = trans ? rowc(be) : colc(be);
      MV vin = sub(Vin, ic);
      MV t;
      t.clus = -1;
      int32_t cap = L_.cap[be];
      int64_t toff = alloc((int64_t)cap * std::max(vin.v.cols, 1));
      t.buf = new_buf_single();
      bind_alloc(t.buf);
      t.v = View{toff, 1, cap, cap, vin.v.cols, vin.v.slot, 0};
      Task k = make(TK_PROJ);
      k.a = A.v;
      k.b = vin.v;
      k.c = t.v;
      begin(k);
      acc(A, false);
      acc(vin, false);
      touch(bufs_[t.buf].seg0, true);
      end();
      T[i] = t;
    }
    // output units: the segment clusters under the out-cluster (or the
    // out-cluster itself when it lies inside one segment)
    units.clear();
    if (seg_end_[oc] - seg_begin_[oc] <= 1) {
      units.push_back(oc);
    } else {
      for (int32_t q = seg_begin_[oc]; q < seg_end_[oc]; ++q) units.push_back(seg_cluster_[q]);
    }
    const int32_t nu = (int32_t)units.size();
    const int32_t u0 = seg_begin_[oc];
    auto unit_of = [&](int32_t segidx) { return nu == 1 ? 0 : segidx - u0; };
    cnt.assign(nu + 1, 0);
    for (size_t i = 0; i < lv.size(); ++i) {
      int32_t obc = trans ? colc(lv[i]) : rowc(lv[i]);
      for (int32_t q = seg_begin_[obc]; q < seg_end_[obc]; ++q) cnt[unit_of(q) + 1]++;
    }
    for (int32_t l = 0; l < nu; ++l) cnt[l + 1] += cnt[l];
    fill.assign(cnt.begin(), cnt.end() - 1);
    items.resize(cnt[nu]);
    for (size_t i = 0; i < lv.size(); ++i) {
      int32_t obc = trans ? colc(lv[i]) : rowc(lv[i]);
      for (int32_t q = seg_begin_[obc]; q < seg_end_[obc]; ++q) items[fill[unit_of(q)]++] = (int32_t)i;
    }
    MV kview = Vin;
    group.resize(items.size());
    for (int32_t l = 0; l < nu; ++l) {
      uint64_t used = overwrite ? 1 : 0;  // groups with a task
      for (int32_t q = cnt[l]; q < cnt[l + 1]; ++q) {
        int g = 0;
        if (late_seg >= 0 && !overwrite)
          for (int32_t dist = late_seg - (seg_end_[colc(lv[items[q]])] - 1); dist > 0; dist >>= 1) ++g;
        group[q] = (int8_t)g;
        used |= uint64_t(1) << g;
      }
      for (int g = 63; g >= 0 && used; --g) {
        if (!(used >> g & 1)) continue;
        used ^= uint64_t(1) << g;
        part.clear();
        for (int32_t q = cnt[l]; q < cnt[l + 1]; ++q)
          if (group[q] == g) part.push_back(items[q]);
        emit_rowmv(lv, T, part, Vin, Vout, units[l], sign, trans, overwrite, out_slot, kview);
      }
    }
  }
  // the terms of a ROWMV task for unit lc, with their reads
  void push_terms(const std::vector<int32_t>& lv, const std::vector<MV>& T, const std::vector<int32_t>& list,
                  const MV& Vin, int32_t lc, bool trans) {
    for (int32_t i : list) {
      int32_t be = lv[i];
      int32_t obc = trans ? colc(be) : rowc(be);
      // the term covers rows (obc intersect lc) of the unit
      int32_t rc = C_[obc].size <= C_[lc].size ? obc : lc;
      Term tm;
      std::memset(&tm, 0, sizeof(tm));
      tm.roff = C_[rc].off - C_[lc].off;
      if (kind(be) == KIND_DENSE) {
        MV A = sub(trans ? mvDT(be) : mvD(be), rc);
        MV Bv = sub(Vin, trans ? rowc(be) : colc(be));
        tm.A = A.v;
        tm.B = Bv.v;
        acc(A, false);
        acc(Bv, false);
      } else {
        MV A = sub(trans ? mvY(be) : mvX(be), rc);
        tm.A = A.v;
        tm.B = T[i].v;
        acc(A, false);
        touch(bufs_[T[i].buf].seg0, false);
      }
      grow4(S_->terms);
      S_->terms.push_back(tm);
    }
  }
  // one ROWMV task: unit lc of Vout (+)= sign * sum over the listed leaves
  void emit_rowmv(const std::vector<int32_t>& lv, const std::vector<MV>& T, const std::vector<int32_t>& list,
                  const MV& Vin, const MV& Vout, int32_t lc, float sign, bool trans, bool overwrite,
                  int32_t out_slot, const MV& kview) {
    {
      Task k = make(TK_ROWMV);
      k.flags = overwrite ? TF_OVERWRITE : 0;
      k.sign = sign;
      k.c = sub(Vout, lc).v;
      k.b = Vin.v;  // column count source
      k.out_slot = out_slot;
      k.list_begin = (int32_t)S_->terms.size();
      k.list_count = (int32_t)list.size();
      begin(k);
      push_terms(lv, T, list, Vin, lc, trans);
      acc_rank(kview);
      acc(sub(Vout, lc), true);
      end();
    }
  }
  MV hmul_new(int32_t b, const MV& Vin, bool trans) {
    int32_t oc = trans ? colc(b) : rowc(b);
    MV out = new_temp(oc, Vin.v.cols);
    hmul(b, Vin, out, 1.0f, trans, true, out.v.slot);
    return out;
  }

  // ---------------------------------------------------------------- triangular
  void solve_lower(int32_t d, const MV& V) {
    if (kind(d) == KIND_DENSE) {
      trsm_leaf(TK_TRSM_L, d, V);
      return;
    }
    const Cluster& c = C_[rowc(d)];
    MV V0 = sub(V, c.son[0]), V1 = sub(V, c.son[1]);
    solve_lower(son(d, 0, 0), V0);
    hmul(son(d, 1, 0), V0, V1, -1.0f, false, false, -1, seg_end_[c.son[0]] - 1);
    solve_lower(son(d, 1, 1), V1);
  }
  void solve_upperT(int32_t d, const MV& W) {
    if (kind(d) == KIND_DENSE) {
      trsm_leaf(TK_TRSM_UT, d, W);
      return;
    }
    const Cluster& c = C_[rowc(d)];
    MV W0 = sub(W, c.son[0]), W1 = sub(W, c.son[1]);
    solve_upperT(son(d, 0, 0), W0);
    hmul(son(d, 0, 1), W0, W1, -1.0f, true, false, -1);
    solve_upperT(son(d, 1, 1), W1);
  }
  // ---------------------------------------------------------------- truncation
  // one piece of a TRUNC or DADD task, with its reads
  void push_piece(const PieceMV& p, bool alpha) {
    Piece q;
    std::memset(&q, 0, sizeof(q));
    q.X = p.p.X.v;
    q.Y = p.p.Y.v;
    q.xoff = p.xoff;
    q.yoff = p.yoff;
    q.sign = p.sign;
    q.pad = (alpha ? PF_ALPHA : 0) | (p.nwin == 0 ? 0 : PF_DENSE);
    for (int32_t b = p.win0; b < p.win0 + p.nwin; ++b) touch(bufs_[b].seg0, false);
    grow4(S_->pieces);
    S_->pieces.push_back(q);
    acc(p.p.X, false);
    acc(p.p.Y, false);
  }
  void emit_trunc(const MV& X, const MV& Y, int32_t slot, int32_t cap,
                  const std::vector<PieceMV>& ps, bool alpha = false) {
    Task t = make(TK_TRUNC);
    t.a = X.v;
    t.b = Y.v;
    t.out_slot = slot;
    t.cap = cap;
    t.list_begin = (int32_t)S_->pieces.size();
    t.list_count = (int32_t)ps.size();
    int32_t W = 0;
    begin(t);
    for (const PieceMV& p : ps) {
      push_piece(p, alpha);
      W += p.p.X.v.cols;
    }
    acc(X, true);
    acc(Y, true);
    end();
    L_.wmax = std::max(L_.wmax, W);
    L_.max_trunc_rows = std::max(L_.max_trunc_rows, std::max(X.v.rows, Y.v.rows));
  }
  // Ends of the batches of n pieces, oldest first: the short one comes first
  // (ending with one or two pieces, n = 24 took 837 ms instead of 709 ms).
  // Updates that are not accumulated are truncated whole.
  std::vector<size_t> batches(size_t n) const {
    const size_t most = accumulate_ ? kBatch : std::max<size_t>(n, 1);
    std::vector<size_t> ends;
    for (size_t q = n % most ? n % most : most; q < n; q += most) ends.push_back(q);
    ends.push_back(n);
    return ends;
  }
  bool small_target(int32_t rc, int32_t cc) const {
    return sz(rc) <= kOneStepAgglomeration && sz(cc) <= kOneStepAgglomeration;
  }
  // Many updates of a small target are summed densely before one truncation:
  // one chain of DADD tasks per 64 x 64 window, the newest pieces last, so that
  // the piece completing the sum has little work behind it.  Returns the sum
  // as one piece.
  PieceMV dense_sum(int32_t rc, int32_t cc, const std::vector<PieceMV>& ps) {
    constexpr int32_t kWindow = 64;
    const int32_t m = sz(rc), n = sz(cc);
    PieceMV out;
    out.xoff = out.yoff = 0;
    out.sign = 1.0f;
    const int64_t off = alloc((int64_t)m * n);
    out.p.X.buf = -1;  // tracked per window
    out.p.X.clus = rc;
    out.p.X.at = last_alloc_pos_;
    out.p.X.v = View{off, 1, m, m, n, -1, 0};
    out.p.Y = mvIdent(cc);
    const std::vector<int32_t> fences = pending_fence_;
    for (int32_t wi = 0; wi < m; wi += kWindow)
      for (int32_t wj = 0; wj < n; wj += kWindow) {
        pending_fence_ = fences;
        const int32_t buf = new_buf_single();
        bind_alloc(buf);
        if (out.nwin++ == 0) out.win0 = buf;
        const int32_t wm = std::min(kWindow, m - wi), wn = std::min(kWindow, n - wj);
        std::vector<const PieceMV*> in;
        for (const PieceMV& p : ps)
          if (p.xoff < wi + wm && p.xoff + p.p.X.v.rows > wi && p.yoff < wj + wn && p.yoff + p.p.Y.v.rows > wj)
            in.push_back(&p);
        for (size_t q0 = 0; q0 < std::max<size_t>(in.size(), 1); q0 += kDenseBatch) {
          Task t = make(TK_DADD);
          t.flags = TF_PIECES | (q0 == 0 ? TF_OVERWRITE : 0);
          t.c = View{off + wi + (int64_t)wj * m, 1, m, wm, wn, -1, 0};
          t.a.rows = wi;
          t.a.cols = wj;
          t.list_begin = (int32_t)S_->pieces.size();
          begin(t);
          for (size_t q = q0; q < std::min(in.size(), q0 + kDenseBatch); ++q) push_piece(*in[q], false);
          S_->tasks.back().list_count = (int32_t)S_->pieces.size() - t.list_begin;
          touch(bufs_[buf].seg0, true);
          end();
        }
      }
    return out;
  }
  LR trunc_new(int32_t rc, int32_t cc, const std::vector<PieceMV>& ps) {
    int32_t cap = std::min(kcap_, std::min(sz(rc), sz(cc)));
    int32_t slot = new_slot();
    LR r;
    r.X.clus = rc;
    int64_t xo = alloc((int64_t)sz(rc) * cap);
    r.X.at = last_alloc_pos_;
    r.X.buf = new_buf_leaves(rc);
    bind_alloc(r.X.buf);
    r.X.v = View{xo, 1, sz(rc), sz(rc), cap, slot, 0};
    r.Y.clus = cc;
    int64_t yo = alloc((int64_t)sz(cc) * cap);
    r.Y.at = last_alloc_pos_;
    r.Y.buf = new_buf_leaves(cc);
    bind_alloc(r.Y.buf);
    r.Y.v = View{yo, 1, sz(cc), sz(cc), cap, slot, 0};
    if (accumulate_ && small_target(rc, cc) && ps.size() > kDirect) {
      emit_trunc(r.X, r.Y, slot, cap, {dense_sum(rc, cc, ps)});
      return r;
    }
    const std::vector<size_t> ends = batches(ps.size());
    for (size_t k = 0, q0 = 0; k < ends.size(); q0 = ends[k++]) {
      std::vector<PieceMV> batch;
      if (q0 > 0) batch.push_back(PieceMV{r, 0, 0, 1.0f});
      batch.insert(batch.end(), ps.begin() + q0, ps.begin() + ends[k]);
      emit_trunc(r.X, r.Y, slot, cap, batch);
    }
    return r;
  }

  // ---------------------------------------------------------------- H-gemm
  // X Y^T = the product of blocks a and b that are not both subdivided: exact
  // factors, of the narrowest width for two dense blocks
  LR product(int32_t a, int32_t b) {
    int32_t ka = kind(a), kb = kind(b);
    int32_t tau = rowc(a), sig = colc(a), rho = colc(b);
    if (ka == KIND_ADM) return LR{mvX(a), hmul_new(b, mvY(a), true)};
    if (kb == KIND_ADM) return LR{hmul_new(a, mvX(b), false), mvY(b)};
    if (ka == KIND_DENSE && kb == KIND_DENSE) {
      // exact factors of the narrowest width among |sigma|, |tau|, |rho|
      int32_t ws = sz(sig), wt = sz(tau), wr = sz(rho);
      if (ws <= kcap_ || (ws <= wt && ws <= wr)) return LR{mvD(a), mvDT(b)};
      MV P = new_dense_temp(tau, sz(rho));
      Task t = make(TK_DADD);
      t.flags = TF_OVERWRITE;
      t.c = P.v;
      t.a = mvD(a).v;
      t.b = mvDT(b).v;
      begin(t);
      acc(mvD(a), false);
      acc(mvDT(b), false);
      acc(P, true);
      end();
      if (wr <= wt) return LR{P, mvIdent(rho)};
      // P^T as the Y factor: rows rho, columns |tau|
      MV PT = P;
      PT.clus = rho;
      PT.v = View{P.v.off, sz(tau), 1, sz(rho), sz(tau), -1, 0};
      return LR{mvIdent(tau), PT};
    }
    if (ka == KIND_DENSE) return LR{mvIdent(tau), hmul_new(b, mvDT(a), true)};
    return LR{hmul_new(a, mvD(b), false), mvIdent(rho)};
  }
  // X Y^T = the product of any two blocks, two subdivided ones agglomerated:
  // the eight son products in one truncation for a small target, else two per
  // quadrant (four independent tasks) and then the four quadrants.
  LR product_any(int32_t a, int32_t b) {
    if (!both_sub(a, b)) return product(a, b);
    const Cluster& T = C_[rowc(a)];
    const Cluster& R = C_[colc(b)];
    const bool one_step = small_target(rowc(a), colc(b));
    std::vector<PieceMV> ps;
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < 2; ++j) {
        const int32_t ts = T.son[i], rs = R.son[j], xo = C_[ts].off - T.off, yo = C_[rs].off - R.off;
        std::vector<PieceMV> q;
        for (int k = 0; k < 2; ++k) q.push_back(PieceMV{product_any(son(a, i, k), son(b, k, j)), 0, 0, 1.0f});
        if (!one_step) q = {PieceMV{trunc_new(ts, rs, q), 0, 0, 1.0f}};
        for (PieceMV& p : q) {
          p.xoff = xo;
          p.yoff = yo;
          ps.push_back(p);
        }
      }
    return trunc_new(rowc(a), colc(b), ps);
  }
  bool both_sub(int32_t a, int32_t b) const { return kind(a) == KIND_SUB && kind(b) == KIND_SUB; }
  typedef std::vector<std::pair<int32_t, int32_t>> Pairs;

  // The products of several block pairs with target tau x rho, as pieces at
  // (xoff, yoff): exact factors where one block is not subdivided.  Subdivided
  // pairs are agglomerated together: their son products for a small target,
  // else quadrant by quadrant, every pair's son products of a quadrant
  // summed and truncated at once (four independent tasks).
  void eval_pairs(int32_t tau, int32_t rho, const Pairs& ab, int32_t xoff, int32_t yoff, float sign,
                  std::vector<PieceMV>& out) {
    Pairs subs;
    for (const auto& q : ab)
      if (both_sub(q.first, q.second))
        subs.push_back(q);
      else
        out.push_back(PieceMV{product(q.first, q.second), xoff, yoff, sign});
    if (subs.empty()) return;
    const Cluster& T = C_[tau];
    const Cluster& R = C_[rho];
    const bool one_step = small_target(tau, rho);
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < 2; ++j) {
        const int32_t ts = T.son[i], rs = R.son[j], xo = xoff + C_[ts].off - T.off, yo = yoff + C_[rs].off - R.off;
        Pairs sons;
        for (const auto& q : subs)
          for (int k = 0; k < 2; ++k) sons.emplace_back(son(q.first, i, k), son(q.second, k, j));
        if (one_step) {
          eval_pairs(ts, rs, sons, xo, yo, sign, out);
          continue;
        }
        std::vector<PieceMV> ps;
        eval_pairs(ts, rs, sons, 0, 0, 1.0f, ps);
        out.push_back(PieceMV{trunc_new(ts, rs, ps), xo, yo, sign});
      }
  }

  // c <- c + sign * sum_p X_p Y_p^T in the format of c, a leaf, in batches
  // (sums: small targets may sum many pieces densely first, which allocates)
  void add_pieces(int32_t c, const std::vector<PieceMV>& ps, bool sums = true) {
    if (kind(c) == KIND_DENSE) {
      for (size_t q0 = 0; q0 < ps.size(); q0 += kDenseBatch) {
        Task t = make(TK_DADD);
        t.flags = TF_PIECES;
        t.c = mvD(c).v;
        t.list_begin = (int32_t)S_->pieces.size();
        begin(t);
        for (size_t q = q0; q < std::min(ps.size(), q0 + kDenseBatch); ++q) push_piece(ps[q], false);
        S_->tasks.back().list_count = (int32_t)S_->pieces.size() - t.list_begin;
        acc(mvD(c), true);
        end();
      }
      return;
    }
    if (sums && accumulate_ && small_target(rowc(c), colc(c)) && ps.size() > kDirect) {
      const PieceMV sum = dense_sum(rowc(c), colc(c), ps);
      emit_trunc(mvX(c), mvY(c), L_.slot[c], L_.cap[c], {PieceMV{LR{mvX(c), mvY(c)}, 0, 0, 1.0f}, sum});
      return;
    }
    if (ps.empty()) return;
    const std::vector<size_t> ends = batches(ps.size());
    for (size_t k = 0, q0 = 0; k < ends.size(); q0 = ends[k++]) {
      std::vector<PieceMV> batch;
      batch.push_back(PieceMV{LR{mvX(c), mvY(c)}, 0, 0, 1.0f});
      batch.insert(batch.end(), ps.begin() + q0, ps.begin() + ends[k]);
      emit_trunc(mvX(c), mvY(c), L_.slot[c], L_.cap[c], batch);
    }
  }

  // c <- c + sign * a b in the format of c (the H-LU's Schur complement update
  // is sign = -1).
  // Accumulated: the update is noted at c and moves down the block tree when c
  // is used (settle), so that a leaf receives the updates of all steps and
  // levels together and truncates their sum in batches.  At n = 24 that is 0.19
  // M truncations and 0.70 M dense updates instead of 1.14 M and 4.7 M.
  // Otherwise every product is formed at the largest block it has and added at
  // once, down to the leaves, each of which truncates it.
  void gemm(int32_t c, int32_t a, int32_t b, float sign = -1.0f) {
    if (!accumulate_) {
      gemm_at_once(c, a, b, sign);
      return;
    }
    Update u;
    u.a = a;
    u.b = b;
    u.sign = sign;
    note_update(c, u);
  }
  void gemm_at_once(int32_t c, int32_t a, int32_t b, float sign) {
    if (kind(c) != KIND_SUB || !both_sub(a, b)) {
      add_products(c, {product_any(a, b)}, sign);
      return;
    }
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < 2; ++j) {
        // the two son products into c_ij that are not themselves subdivided
        // products are added together
        const int32_t cc = son(c, i, j);
        std::vector<LR> ps;
        for (int k = 0; k < 2; ++k) {
          const int32_t aa = son(a, i, k), bb = son(b, k, j);
          if (kind(cc) == KIND_SUB && both_sub(aa, bb))
            gemm_at_once(cc, aa, bb, sign);
          else
            ps.push_back(product_any(aa, bb));
        }
        add_products(cc, ps, sign);
      }
  }
  void add_products(int32_t c, const std::vector<LR>& ps, float sign) {
    std::vector<PieceMV> pieces;
    for (const LR& p : ps) pieces.push_back(PieceMV{p, 0, 0, sign});
    if (!pieces.empty()) add_down(c, pieces);
  }
  // The updates noted at c, before c is factored, solved or read: a leaf adds
  // them, a subdivided block hands them to its sons (products that are not
  // subdivided x subdivided are formed here, at c's size).
  void settle(int32_t c) {
    std::vector<Update> us;
    us.swap(updates_[c]);
    if (us.empty()) return;
    std::sort(us.begin(), us.end(), [](const Update& x, const Update& y) { return x.seq < y.seq; });
    if (kind(c) != KIND_SUB) {
      // low-rank updates exist already; they and the products below are added
      // early when forming a product would come close to reusing their memory
      std::vector<std::pair<int64_t, PieceMV>> got;
      Pairs subs;
      const float sign = us[0].sign;
      int64_t least = kNotTemp;  // position of the oldest factor
      for (const Update& u : us) {
        if (u.sign != sign) throw std::logic_error("updates of one block with different signs");
        if (u.a >= 0) continue;
        got.emplace_back(u.seq, PieceMV{u.p, 0, 0, sign});
        least = std::min(least, position(u.p));
      }
      auto add = [&]() {
        std::stable_sort(got.begin(), got.end(),
                         [](const std::pair<int64_t, PieceMV>& x, const std::pair<int64_t, PieceMV>& y) {
                           return x.first < y.first;
                         });
        std::vector<PieceMV> ps;
        for (auto& g : got) ps.push_back(g.second);
        add_pieces(c, ps);
        got.clear();
        least = kNotTemp;
      };
      for (const Update& u : us) {
        if (u.a < 0) continue;
        if (both_sub(u.a, u.b)) {
          subs.emplace_back(u.a, u.b);
          continue;
        }
        if (least != kNotTemp && least + ring_size_ - ring_pos() < ring_size_ / 8) add();
        got.emplace_back(u.seq, PieceMV{product(u.a, u.b), 0, 0, sign});
        least = std::min(least, position(got.back().second.p));
      }
      std::vector<PieceMV> ps;
      if (!subs.empty()) {
        if (least != kNotTemp && least + ring_size_ - ring_pos() < ring_size_ / 8) add();
        eval_pairs(rowc(c), colc(c), subs, 0, 0, sign, ps);
      }
      // the agglomerated pairs after the rest
      for (const PieceMV& q : ps) got.emplace_back(INT64_MAX, q);
      add();
      return;
    }
    // what exists first: the products formed below may reuse ring memory
    for (int pass = 0; pass < 2; ++pass)
      for (Update& u : us) {
        if ((u.a >= 0) != (pass == 1)) continue;
        if (u.a >= 0 && both_sub(u.a, u.b)) {
          for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j)
              for (int k = 0; k < 2; ++k) {
                Update v = u;
                v.a = son(u.a, i, k);
                v.b = son(u.b, k, j);
                note_update(son(c, i, j), v, u.seq);
              }
          continue;
        }
        Update v = u;
        if (u.a >= 0) v.p = product(u.a, u.b);
        v.a = v.b = -1;
        const LR p = v.p;
        for (int i = 0; i < 2; ++i)
          for (int j = 0; j < 2; ++j) {
            v.p = LR{sub(p.X, C_[rowc(c)].son[i]), sub(p.Y, C_[colc(c)].son[j])};
            note_update(son(c, i, j), v, u.seq);
          }
      }
  }
  void settle_all(int32_t c) {
    settle(c);
    if (kind(c) == KIND_SUB)
      for (int k = 0; k < 4; ++k) settle_all(B_[c].son[k]);
  }

  // ---------------------------------------------------------------- whole H-matrices
  // dst <- sign * src (times the launch's alpha when `alpha`), leaf by leaf;
  // dst and src have the same block structure.  Dense leaves: one DADD of
  // src against the identity; admissible leaves: a truncation of the one
  // piece (exact: the rank does not change).
  void copy_scaled(int32_t dst, int32_t src, float sign, bool alpha) {
    if (kind(dst) == KIND_SUB) {
      for (int k = 0; k < 4; ++k) copy_scaled(B_[dst].son[k], B_[src].son[k], sign, alpha);
      return;
    }
    if (kind(dst) == KIND_DENSE) {
      // dense blocks have one side of at most a tile: D I or I D
      Task t = make(TK_DADD);
      t.flags = TF_OVERWRITE | (alpha ? TF_ALPHA : 0);
      t.sign = sign;
      t.c = mvD(dst).v;
      if (sz(colc(dst)) <= sz(rowc(dst))) {
        t.a = mvD(src).v;
        t.b = mvIdent(colc(dst)).v;
      } else {
        t.a = mvIdent(rowc(dst)).v;
        t.b = mvDT(src).v;
      }
      begin(t);
      acc(mvD(src), false);
      acc(mvD(dst), true);
      end();
      return;
    }
    PieceMV p{LR{mvX(src), mvY(src)}, 0, 0, sign};
    std::vector<PieceMV> ps{p};
    emit_trunc(mvX(dst), mvY(dst), L_.slot[dst], L_.cap[dst], ps, alpha);
  }
  // dst <- 0: dense leaves overwritten with an empty product, admissible
  // leaves truncated from no pieces (rank 0)
  void zero(int32_t dst) {
    if (kind(dst) == KIND_SUB) {
      for (int k = 0; k < 4; ++k) zero(B_[dst].son[k]);
      return;
    }
    if (kind(dst) == KIND_DENSE) {
      Task t = make(TK_DADD);
      t.flags = TF_OVERWRITE;
      t.c = mvD(dst).v;
      t.a = mvD(dst).v;
      t.a.cols = 0;  // no columns: the product is zero
      t.b = mvDT(dst).v;
      t.b.cols = 0;
      begin(t);
      acc(mvD(dst), true);
      end();
      return;
    }
    emit_trunc(mvX(dst), mvY(dst), L_.slot[dst], L_.cap[dst], {});
  }
  // Vout <- H(b) Vin for a whole H-matrix b (its row cluster is the root)
  void apply(int32_t b, const MV& Vin, const MV& Vout) { hmul(b, Vin, Vout, 1.0f, false, true, Vout.v.slot); }

  // ---------------------------------------------------------------- H-trsm, H-LU
  void trsm_left(int32_t d, int32_t b) {
    settle(b);
    int32_t k = kind(b);
    if (k == KIND_ADM) {
      solve_lower(d, mvX(b));
    } else if (k == KIND_DENSE) {
      solve_lower(d, mvD(b));
    } else {
      for (int j = 0; j < 2; ++j) {
        trsm_left(son(d, 0, 0), son(b, 0, j));
        gemm(son(b, 1, j), son(d, 1, 0), son(b, 0, j));
        trsm_left(son(d, 1, 1), son(b, 1, j));
      }
    }
  }
  void trsm_right(int32_t b, int32_t d) {
    settle(b);
    int32_t k = kind(b);
    if (k == KIND_ADM) {
      solve_upperT(d, mvY(b));
    } else if (k == KIND_DENSE) {
      solve_upperT(d, mvDT(b));
    } else {
      for (int i = 0; i < 2; ++i) {
        trsm_right(son(b, i, 0), son(d, 0, 0));
        gemm(son(b, i, 1), son(b, i, 0), son(d, 0, 1));
        trsm_right(son(b, i, 1), son(d, 1, 1));
      }
    }
  }
  void lu(int32_t d) {
    settle(d);
    if (kind(d) == KIND_DENSE) {
      getrf(d);
      return;
    }
    int32_t d00 = son(d, 0, 0), d01 = son(d, 0, 1), d10 = son(d, 1, 0), d11 = son(d, 1, 1);
    lu(d00);
    trsm_left(d00, d01);
    trsm_right(d10, d00);
    gemm(d11, d10, d01);
    lu(d11);
  }

  // ---------------------------------------------------------------- the solve of step III
  // x = U^-1 (L^-1 P w).  The chain through the diagonal runs over solve
  // blocks (clusters of up to kSolveBlock DOFs) instead of tiles: a block is
  // one parallel step, its units multiplied by their row panels of the
  // inverted triangular factor (overwriting ROWMV tasks).  w and x share the
  // work vector, the forward result has its own (z).
  void solve_all(int32_t nrhs_max) {
    const int32_t N = sz(0);
    W_.buf = new_buf_leaves(0);  // per-segment tracking over the whole vector
    Z_.buf = new_buf_leaves(0);
    W_.clus = Z_.clus = 0;
    W_.v = View{L_.work_off, 1, N, N, nrhs_max, L_.nrhs_slot, 0};
    Z_.v = View{L_.z_off, 1, N, N, nrhs_max, L_.nrhs_slot, 0};
    // the unit (diagonal tile) and the block of every segment, by offset
    blk_of_seg_.clear();
    unit_of_seg_.clear();
    size_t u = 0;
    int32_t end = L_.inv_units[0].rows, blk = 0;  // end of unit u in the whole vector
    for (int32_t q : seg_cluster_) {
      while (C_[q].off >= end) {
        ++u;
        end += L_.inv_units[u].rows;
        if (L_.inv_units[u].first == (int32_t)u) ++blk;
      }
      if (C_[q].off + sz(q) > end) throw std::logic_error("a segment crosses a diagonal tile");
      unit_of_seg_.push_back((int32_t)u);
      blk_of_seg_.push_back(blk);
    }
    solve_diag(0, true);
    solve_diag(0, false);
  }
  void solve_diag(int32_t d, bool fwd) {
    const Cluster& c = C_[rowc(d)];
    if (kind(d) == KIND_DENSE || c.size <= kSolveBlock) {
      for (int32_t q = seg_begin_[rowc(d)]; q < seg_end_[rowc(d)]; ++q) inv_unit(q, fwd);
      return;
    }
    solve_diag(son(d, fwd ? 0 : 1, fwd ? 0 : 1), fwd);
    solve_update(fwd ? son(d, 1, 0) : son(d, 0, 1), fwd);
    solve_diag(son(d, fwd ? 1 : 0, fwd ? 1 : 0), fwd);
  }
  // one segment's rows of its block's inverse times the block's right-hand side
  void inv_unit(int32_t q, bool fwd) {
    const InvUnit& u = L_.inv_units[unit_of_seg_[q]];
    const MV& in = fwd ? W_ : Z_;
    const MV out = sub(fwd ? Z_ : W_, seg_cluster_[q]);
    // input: the block up to the unit's end, or from its start on
    int32_t s0 = q, s1 = q + 1;
    while (s0 > 0 && (fwd ? blk_of_seg_[s0 - 1] == blk_of_seg_[q] : unit_of_seg_[s0 - 1] == unit_of_seg_[q])) --s0;
    while (s1 < (int32_t)seg_cluster_.size() &&
           (fwd ? unit_of_seg_[s1] == unit_of_seg_[q] : blk_of_seg_[s1] == blk_of_seg_[q]))
      ++s1;
    const int32_t cols = fwd ? u.begin + u.rows : u.m - u.begin;
    const int32_t in0 = C_[seg_cluster_[s0]].off, row = C_[seg_cluster_[q]].off - (fwd ? in0 + u.begin : in0);
    Term tm;
    std::memset(&tm, 0, sizeof(tm));
    tm.A = View{(fwd ? u.l_off : u.u_off) + row, 1, u.ld, out.v.rows, cols, -1, 0};
    tm.B = in.v;
    tm.B.off += in0;
    tm.B.rows = cols;
    Task k = make(TK_ROWMV);
    k.flags = TF_OVERWRITE;
    k.c = out.v;
    k.b = in.v;  // column count source
    k.list_begin = (int32_t)S_->terms.size();
    k.list_count = 1;
    grow4(S_->terms);
    S_->terms.push_back(tm);
    begin(k);
    for (int32_t s = s0; s < s1; ++s) acc(sub(in, seg_cluster_[s]), false);
    acc(out, true);
    end();
  }
  // out -= H(b) in for an off-diagonal block, in solved before out.  Terms and
  // projections are grouped by how many solve blocks before the last one of
  // the input they are final (group 0 the last block, group g blocks 2^(g-1)
  // to 2^g - 1 before it) and run far groups first, so that little work
  // waits for the last block.  Output units solved kMergeBlocks or more blocks
  // later have time: all their terms go into one task.
  void solve_update(int32_t b, bool fwd) {
    constexpr int32_t kMergeBlocks = 2;
    const MV in = sub(fwd ? Z_ : W_, colc(b)), out = sub(fwd ? W_ : Z_, rowc(b));
    std::vector<int32_t> lv;
    leaves_of(b, lv);
    const int32_t last = fwd ? blk_of_seg_[seg_end_[colc(b)] - 1] : blk_of_seg_[seg_begin_[colc(b)]];
    auto group = [&](int32_t seg) {
      int g = 0;
      for (int32_t dist = std::abs(blk_of_seg_[seg] - last); dist > 0; dist >>= 1) ++g;
      return g;
    };
    std::vector<MV> T(lv.size());
    for (size_t i = 0; i < lv.size(); ++i) {
      const int32_t be = lv[i];
      if (kind(be) != KIND_ADM) continue;
      const MV A = mvY(be), vin = sub(in, colc(be));
      const int32_t cap = L_.cap[be];
      MV t;
      t.clus = -1;
      const int64_t toff = alloc((int64_t)cap * std::max(vin.v.cols, 1));
      t.buf = new_buf_single();
      bind_alloc(t.buf);
      t.v = View{toff, 1, cap, cap, vin.v.cols, vin.v.slot, 0};
      // one task per run of segments of the same group, the farthest first
      const int32_t s0 = seg_begin_[colc(be)], s1 = seg_end_[colc(be)];
      bool add = false;
      for (int32_t done = 0; done < s1 - s0;) {
        int32_t n = 1;
        auto at = [&](int32_t k) { return fwd ? s0 + k : s1 - 1 - k; };
        while (done + n < s1 - s0 && group(at(done + n)) == group(at(done))) ++n;
        const int32_t lo = std::min(at(done), at(done + n - 1)), hi = lo + n;
        const bool whole = n == s1 - s0;  // (a column cluster inside one segment has no segment of its own)
        const int32_t r0 = whole ? 0 : C_[seg_cluster_[lo]].off - C_[colc(be)].off;
        const int32_t r1 = whole ? sz(colc(be))
                                 : C_[seg_cluster_[hi - 1]].off + sz(seg_cluster_[hi - 1]) - C_[colc(be)].off;
        Task k = make(TK_PROJ);
        k.flags = add ? TF_ADD : 0;
        k.a = A.v;
        k.b = vin.v;
        k.c = t.v;
        k.a.off += r0;
        k.b.off += r0;
        k.a.rows = k.b.rows = r1 - r0;
        begin(k);
        if (whole)
          acc(vin, false);
        else
          for (int32_t s = lo; s < hi; ++s) acc(sub(in, seg_cluster_[s]), false);
        touch(bufs_[t.buf].seg0, true);
        end();
        add = true;
        done += n;
      }
      T[i] = t;
    }
    const int32_t u0 = seg_begin_[rowc(b)], nu = seg_end_[rowc(b)] - u0;
    std::vector<std::vector<int32_t>> items(nu);
    for (size_t i = 0; i < lv.size(); ++i)
      for (int32_t q = seg_begin_[rowc(lv[i])]; q < seg_end_[rowc(lv[i])]; ++q) items[q - u0].push_back((int32_t)i);
    const int32_t first = fwd ? blk_of_seg_[u0] : blk_of_seg_[u0 + nu - 1];
    constexpr int kGroups = 33;
    for (int32_t l = 0; l < nu; ++l) {
      const int32_t unit = nu == 1 ? rowc(b) : seg_cluster_[u0 + l];
      const bool merge = std::abs(blk_of_seg_[u0 + l] - first) >= kMergeBlocks;
      std::vector<int32_t> parts[kGroups];
      for (int32_t i : items[l]) {
        const int32_t ic = colc(lv[i]);
        parts[merge ? 0 : group(fwd ? seg_end_[ic] - 1 : seg_begin_[ic])].push_back(i);
      }
      for (int g = kGroups - 1; g >= 0; --g)
        if (!parts[g].empty()) emit_rowmv(lv, T, parts[g], in, out, unit, -1.0f, false, false, -1, in);
    }
  }

 private:
  const std::vector<Cluster>& C_;
  const std::vector<Block>& B_;
  int32_t kcap_;
  ArenaLayout& L_;
  Schedule* S_;
  std::vector<int32_t>& dbuf_;
  std::vector<int32_t>& xbuf_;
  std::vector<int32_t>& ybuf_;
  int32_t segsz_ = 0;
  int64_t ring_off_ = 0, ring_size_ = 0, cursor_ = 0;
  bool accumulate_;
  std::vector<int32_t> seg_begin_, seg_end_, seg_cluster_;
  std::vector<std::vector<int32_t>> chunk_occ_;
  std::vector<int32_t> chunk_fence_task_;
  std::vector<int32_t> chunk_pass_;
  int32_t pass_ = 0;
 public:
  int64_t wraps_ = 0;
  int64_t early_pieces_ = 0;  // pieces that add_old_pieces added
 private:
  std::vector<std::vector<Update>> updates_;                     // per block
  std::unordered_map<int64_t, std::vector<int32_t>> held_;        // per ring bucket: blocks with updates there
  int64_t forced_bucket_ = -kBuckets, update_seq_ = 0;
  std::vector<int32_t> pending_fence_;
  int64_t last_alloc_lo_ = 0, last_alloc_hi_ = -1, last_alloc_pos_ = 0;
  std::vector<int32_t> fence_pool_;
  std::vector<int32_t> acc_task_;
  std::vector<int64_t> acc_next_;
  std::vector<Buf> bufs_;
  std::vector<Seg> segs_;
  std::vector<int32_t> rtask_;
  std::vector<int64_t> rnext_;
  std::vector<int32_t> stamp_, implied_;
  std::vector<int32_t> deps_;
  int32_t cur_ = -1;
  struct {
    std::vector<int32_t> leaves, units, cnt, fill, items, part;
    std::vector<MV> T;
    std::vector<int8_t> group;
  } hm_;                            // hmul's
  MV W_, Z_;                        // the solve's work vector and forward result
  std::vector<int32_t> blk_of_seg_, unit_of_seg_;  // solve block and diagonal tile of each segment
};

}  // namespace

std::vector<Block> factor_tree(const std::vector<Cluster>& C, const std::vector<Block>& B, int32_t tile) {
  std::vector<Block> out;
  out.reserve(B.size());
  // DFS over the block tree; a node whose row and column clusters both hold at
  // most `tile` DOFs becomes one dense tile (its sub-blocks merged exactly)
  struct Rec {
    static int32_t go(const std::vector<Cluster>& C, const std::vector<Block>& B, int32_t tile, int32_t b,
                      int32_t parent, std::vector<Block>& out) {
      const Block& src = B[b];
      int32_t id = (int32_t)out.size();
      out.push_back(src);
      Block& nb = out.back();
      nb.parent = parent;
      for (int k = 0; k < 4; ++k) nb.son[k] = -1;
      int32_t big = std::max(C[src.row].size, C[src.col].size);
      int32_t small = std::min(C[src.row].size, C[src.col].size);
      // a subdivided node turns dense as soon as one of its clusters is a tile,
      // so a dense diagonal tile never meets a subdivided block in its block
      // row or column; an admissible node turns dense when both clusters are
      if ((src.kind == KIND_SUB && small <= tile) || (src.kind == KIND_ADM && big <= tile)) {
        out[id].kind = KIND_DENSE;
        return id;
      }
      if (src.kind == KIND_SUB) {
        int32_t sons[4];
        for (int k = 0; k < 4; ++k) sons[k] = go(C, B, tile, src.son[k], id, out);
        for (int k = 0; k < 4; ++k) out[id].son[k] = sons[k];
      }
      return id;
    }
  };
  Rec::go(C, B, tile, 0, -1, out);
  return out;
}

namespace {

// The solve blocks (diagonal blocks of up to kSolveBlock DOFs, or single
// tiles) with the storage of their inverses; d_off and dst are relative to the
// scratch.  Returns the scratch's size.
template <class Alloc>
int64_t plan_inverses(const std::vector<Cluster>& C, const std::vector<Block>& B, ArenaLayout& L, Alloc& alloc) {
  int64_t scratch = 0;
  struct Rec {
    const std::vector<Cluster>& C;
    const std::vector<Block>& B;
    ArenaLayout& L;
    Alloc& alloc;
    int64_t& scratch;
    void leaves(int32_t b, int32_t off, int32_t ld, int64_t d0) {
      const Block& k = B[b];
      if (k.kind == KIND_SUB) {
        for (int32_t s : k.son) leaves(s, off, ld, d0);
        return;
      }
      InvLeaf f;
      f.dst = d0 + (C[k.row].off - off) + (int64_t)(C[k.col].off - off) * ld;
      f.m = C[k.row].size;
      f.n = C[k.col].size;
      f.ld = ld;
      f.slot = k.kind == KIND_ADM ? L.slot[b] : -1;
      f.off = k.kind == KIND_ADM ? L.x_off[b] : L.dense_off[b];
      f.off2 = k.kind == KIND_ADM ? L.y_off[b] : -1;
      L.inv_leaves.push_back(f);
    }
    void units(int32_t b, int32_t off, int32_t m, int64_t d0) {
      const Block& k = B[b];
      if (k.kind == KIND_SUB) {
        units(k.son[0], off, m, d0);
        units(k.son[3], off, m, d0);
        return;
      }
      InvUnit u;
      u.d_off = d0;
      u.piv_off = L.piv_off[b];
      u.begin = C[k.row].off - off;
      u.rows = C[k.row].size;
      u.m = m;
      u.ld = (u.rows + 3) & ~3;
      u.l_off = alloc((int64_t)u.ld * (u.begin + u.rows));
      u.u_off = alloc((int64_t)u.ld * (m - u.begin));
      L.inv_units.push_back(u);
    }
    void go(int32_t b) {
      const Block& k = B[b];
      const int32_t m = C[k.row].size;
      if (k.kind == KIND_SUB && m > kSolveBlock) {
        go(k.son[0]);
        go(k.son[3]);
        return;
      }
      const int32_t first = (int32_t)L.inv_units.size();
      const int64_t d0 = scratch;
      scratch += ((int64_t)m * m + 31) & ~int64_t(31);
      leaves(b, C[k.row].off, m, d0);
      units(b, C[k.row].off, m, d0);
      for (size_t q = first; q < L.inv_units.size(); ++q) {
        L.inv_units[q].first = first;
        L.inv_units[q].count = (int32_t)L.inv_units.size() - first;
      }
    }
  };
  Rec r{C, B, L, alloc, scratch};
  r.go(0);
  return scratch;
}

// Renumbers the solve's tasks in the order in which a list scheduling with
// kWorkers workers starts them (priority: the longest path to the end), the
// order in which the solve kernel hands them out.  Every task starts after its
// predecessors ended, so the order is topological.  The durations are rough
// (microseconds): a hop and the time to read the operands.
void order_for_tickets(Schedule& S) {
  constexpr int kWorkers = 512;
  const int64_t n = (int64_t)S.tasks.size();
  if (n < 2) return;
  std::vector<float> dur(n), prio(n, 0.0f);
  for (int64_t t = 0; t < n; ++t) {
    const Task& k = S.tasks[t];
    float elems = 0;
    if (k.type == TK_PROJ)
      elems = (float)k.a.rows * std::min(k.a.cols, 12);
    else
      for (int32_t q = 0; q < k.list_count; ++q) {
        const View& A = S.terms[k.list_begin + q].A;
        elems += (float)A.rows * (A.slot >= 0 ? std::min(A.cols, 12) : A.cols);
      }
    dur[t] = 3.0f + elems * 1e-4f;
  }
  std::vector<int64_t> sp(n + 1, 0);
  std::vector<int32_t> si(S.pred_idx.size()), left(n);
  for (int64_t t = 0; t < n; ++t) {
    left[t] = (int32_t)(S.pred_ptr[t + 1] - S.pred_ptr[t]);
    for (int64_t e = S.pred_ptr[t]; e < S.pred_ptr[t + 1]; ++e) ++sp[S.pred_idx[e] + 1];
  }
  for (int64_t t = 0; t < n; ++t) sp[t + 1] += sp[t];
  std::vector<int64_t> fill(sp.begin(), sp.end() - 1);
  for (int64_t t = 0; t < n; ++t)
    for (int64_t e = S.pred_ptr[t]; e < S.pred_ptr[t + 1]; ++e) si[fill[S.pred_idx[e]]++] = (int32_t)t;
  for (int64_t t = n - 1; t >= 0; --t) {
    for (int64_t e = sp[t]; e < sp[t + 1]; ++e) prio[t] = std::max(prio[t], prio[si[e]]);
    prio[t] += dur[t];
  }
  typedef std::pair<float, int32_t> Item;
  std::priority_queue<Item> ready;                                              // by priority, then index
  std::priority_queue<Item, std::vector<Item>, std::greater<Item>> running;     // by end time
  for (int64_t t = 0; t < n; ++t)
    if (left[t] == 0) ready.push(Item(prio[t], -(int32_t)t));
  std::vector<int32_t> order;
  order.reserve(n);
  float now = 0;
  while ((int64_t)order.size() < n) {
    while (!ready.empty() && running.size() < kWorkers) {
      const int32_t t = -ready.top().second;
      ready.pop();
      order.push_back(t);
      running.push(Item(now + dur[t], t));
    }
    if (running.empty()) throw std::logic_error("the solve schedule has a cycle");
    const int32_t t = running.top().second;
    now = running.top().first;
    running.pop();
    for (int64_t e = sp[t]; e < sp[t + 1]; ++e)
      if (--left[si[e]] == 0) ready.push(Item(prio[si[e]], -si[e]));
  }
  std::vector<int32_t> rank(n);
  for (int64_t k = 0; k < n; ++k) rank[order[k]] = (int32_t)k;
  std::vector<Task> tasks(n);
  std::vector<int64_t> pp(1, 0);
  std::vector<int32_t> pi;
  pi.reserve(S.pred_idx.size());
  for (int64_t k = 0; k < n; ++k) {
    const int32_t t = order[k];
    tasks[k] = S.tasks[t];
    const size_t at = pi.size();
    for (int64_t e = S.pred_ptr[t]; e < S.pred_ptr[t + 1]; ++e) pi.push_back(rank[S.pred_idx[e]]);
    std::sort(pi.begin() + at, pi.end());
    pp.push_back((int64_t)pi.size());
  }
  S.tasks.swap(tasks);
  S.pred_ptr.swap(pp);
  S.pred_idx.swap(pi);
}

// Builds a schedule with accumulated updates when asked for and, where their
// temporaries exceed the ring, without.
template <class F>
void with_ring(bool accumulate, ArenaLayout& L, const F& build) {
  if (accumulate) {
    const ArenaLayout before = L;
    try {
      build(true);
      return;
    } catch (const RingFull&) {
      L = before;
    }
  }
  build(false);
}

}  // namespace

// Without tiles (tile 0: the block tree's own small leaves) the accumulated
// updates of a leaf are many and make one long chain of truncations: n = 10,
// leaf 16: 517 ms against 63 ms added at once (FP64, n = 8: 1,838 against 118
// ms).  With tiles the two take about the same time at coarse eps (n = 24, FP32,
// eps 1e-4: 713 against 710 ms), and the accumulated factor is the nearer one
// (one apply leaves 2e-3 of the residual against 1e-2, n = 24).  At finer eps the
// sums' spectra are filled with rounding and the wide truncations cost more, the
// more the larger the mesh.  FP32, accumulated against at once: eps 1e-5 n = 13
// 70.8 : 71.6 (with the solve), n = 16 172 : 155, n = 24 1,126 : 901 ms, at
// kappa 16 n = 24 1.62 : 1.07, n = 32 5.83 : 3.53, n = 40 21.0 : 12.3 s; eps 1e-6
// n = 16 374 : 268, n = 24 2,600 : 1,496 ms.  FP64: eps 1e-6 n = 8 65 : 73, n =
// 11 316 : 311 ms; 1e-12 n = 8 73 : 88, n = 11 576 : 521 ms.  (n = 8: N = 3,032;
// 11: 8,261; 13: 13,897; 16: 26,416.)
bool accumulate_updates(int32_t N, int32_t tile, double eps) {
  return tile > 0 && (eps >= 3e-5 || N < 5000 || (eps >= 4e-6 && N < 20000));
}

void build_schedules(const std::vector<Cluster>& C, const std::vector<Block>& Bfull, int32_t rank_cap,
                     int32_t nrhs_max, int32_t tile, ArenaLayout& L,
                     Schedule& factor, Schedule& solve,
                     SchedStats& st, std::vector<Block>* factor_blocks, bool accumulate, int64_t ring_elems) {
  std::vector<Block> Bt = factor_tree(C, Bfull, tile);
  const std::vector<Block>& B = Bt;
  if (factor_blocks) *factor_blocks = Bt;
  auto t0 = std::chrono::steady_clock::now();
  const size_t nb = B.size();
  L = ArenaLayout();
  L.dense_off.assign(nb, -1);
  L.x_off.assign(nb, -1);
  L.y_off.assign(nb, -1);
  L.cap.assign(nb, 0);
  L.slot.assign(nb, -1);
  L.piv_off.assign(nb, -1);
  int32_t leafmax = 0;
  for (const Cluster& c : C)
    if (c.son[0] < 0) leafmax = std::max(leafmax, c.size);
  auto alloc = [&](int64_t n) {
    int64_t o = L.total;
    L.total += (n + 31) & ~int64_t(31);
    return o;
  };
  L.ident_n = std::max(std::max(leafmax, tile), kOneStepAgglomeration);
  L.ident_off = alloc((int64_t)L.ident_n * L.ident_n);
  int64_t fe = 0;
  for (size_t b = 0; b < nb; ++b) {
    int32_t m = C[B[b].row].size, n = C[B[b].col].size;
    if (B[b].kind == KIND_DENSE) {
      L.dense_off[b] = alloc((int64_t)m * n);
      fe += (int64_t)m * n;
      if (B[b].row == B[b].col) {
        L.piv_off[b] = L.piv_total;
        L.piv_total += m;
      }
    } else if (B[b].kind == KIND_ADM) {
      int32_t cap = std::min(rank_cap, std::min(m, n));
      L.cap[b] = cap;
      L.slot[b] = L.n_slots++;
      L.x_off[b] = alloc((int64_t)m * cap);
      L.y_off[b] = alloc((int64_t)n * cap);
      fe += (int64_t)(m + n) * cap;
    }
  }
  L.factor_elems = fe;
  L.nrhs_max = nrhs_max;
  L.nrhs_slot = L.n_slots++;
  L.work_off = alloc((int64_t)C[0].size * nrhs_max);
  L.z_off = alloc((int64_t)C[0].size * nrhs_max);
  const int64_t inv_scratch = plan_inverses(C, B, L, alloc);
  L.wmax = 0;
  // ring region for temporaries (both schedules; they never run concurrently).
  // Every wrap of the ring orders the new occupants of a chunk after all
  // users of its previous ones (FENCE tasks); at rank capacity 64 the
  // temporaries are twice those of capacity 32, and a 2^31-element bound
  // keeps the number of wraps (and fences) of the larger workloads at what a
  // 2^30 bound gave at capacity 32.
  const int64_t ring =
      ring_elems > 0
          ? ring_elems
          : std::max(inv_scratch, std::min<int64_t>(std::max<int64_t>(8 * fe, int64_t(1) << 22), int64_t(1) << 31));
  const int64_t ring_off = alloc(std::max(ring, inv_scratch));
  L.ring_off = ring_off;
  L.ring_size = ring;
  // the dense copies are scratch between the factorisation and the solves:
  // they use the ring's memory
  for (InvUnit& u : L.inv_units) u.d_off += ring_off;
  for (InvLeaf& f : L.inv_leaves) f.dst += ring_off;
  const int32_t segsz = std::max(leafmax, tile);
  factor = Schedule();
  solve = Schedule();
  // the solve's schedule is built beside the factorisation's, from a layout of
  // its own (it adds nothing to it)
  int64_t solve_temps = 0;
  std::future<void> solved = std::async(std::launch::async | std::launch::deferred, [&, LS = L]() mutable {
    // the solve's units are clusters of half a tile: a step of the chain spreads
    // over twice as many SMs as with whole ones (n = 24, 8 columns: 8.4 -> 7.8 ms
    // an apply, FP64 n = 11 5.2 -> 3.5 ms).  Smaller leaves are no units of their
    // own: their edges are many (n = 16: 0.27 M with units of 32, 2.4 M with leaves
    // of 8, 27 M with leaves of 2) and their rows leave lanes idle.
    std::vector<int32_t> dbuf, xbuf, ybuf;
    Sched s(C, B, rank_cap, LS, &solve, dbuf, xbuf, ybuf, true, std::max(leafmax, tile / 2), false, ring_off, ring);
    s.solve_all(nrhs_max);
    solve_temps = s.temp_elems_;
    order_for_tickets(solve);
  });
  std::vector<int32_t> dbuf, xbuf, ybuf;
  // accumulated updates hold factors for longer; where the ring is too small
  // for that, they are added at once
  with_ring(accumulate, L, [&](bool acc) {
    factor = Schedule();
    Sched s(C, B, rank_cap, L, &factor, dbuf, xbuf, ybuf, true, segsz, acc, ring_off, ring);
    s.lu(0);
    st.temp_elems = s.temp_elems_;
    st.ring_wraps = s.wraps_;
    st.early_pieces = s.early_pieces_;
    st.accumulated = acc;
  });
  solved.get();
  st.temp_elems += solve_temps;
  factor.n_edges = (int64_t)factor.pred_idx.size();
  solve.n_edges = (int64_t)solve.pred_idx.size();
  st.n_factor_tasks = (int64_t)factor.tasks.size();
  st.n_solve_tasks = (int64_t)solve.tasks.size();
  st.host_ms =
      std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
}

void build_inverse_schedules(const std::vector<Cluster>& C, const std::vector<Block>& FB, int32_t rank_cap,
                             int32_t nrhs_max, int32_t tile, ArenaLayout& L, std::vector<Block>& Bx,
                             Schedule& start, Schedule& iter, Schedule& apply, SchedStats& st,
                             int64_t ring_elems) {
  auto t0 = std::chrono::steady_clock::now();
  const int32_t nb = (int32_t)FB.size();
  Bx.assign((size_t)4 * nb, Block());
  for (int32_t q = 0; q < 4; ++q)
    for (int32_t b = 0; b < nb; ++b) {
      Block k = FB[b];
      for (int s = 0; s < 4; ++s)
        if (k.son[s] >= 0) k.son[s] += q * nb;
      if (k.parent >= 0) k.parent += q * nb;
      Bx[(size_t)q * nb + b] = k;
    }
  const size_t nx = Bx.size();
  L = ArenaLayout();
  L.dense_off.assign(nx, -1);
  L.x_off.assign(nx, -1);
  L.y_off.assign(nx, -1);
  L.cap.assign(nx, 0);
  L.slot.assign(nx, -1);
  L.piv_off.assign(nx, -1);
  int32_t leafmax = 0;
  for (const Cluster& c : C)
    if (c.son[0] < 0) leafmax = std::max(leafmax, c.size);
  auto alloc = [&](int64_t n) {
    int64_t o = L.total;
    L.total += (n + 31) & ~int64_t(31);
    return o;
  };
  L.ident_n = std::max(std::max(leafmax, tile), kOneStepAgglomeration);
  L.ident_off = alloc((int64_t)L.ident_n * L.ident_n);
  int64_t fe = 0;
  for (size_t b = 0; b < nx; ++b) {
    const int32_t m = C[Bx[b].row].size, n = C[Bx[b].col].size;
    if (Bx[b].kind == KIND_DENSE) {
      L.dense_off[b] = alloc((int64_t)m * n);
      fe += (int64_t)m * n;
    } else if (Bx[b].kind == KIND_ADM) {
      const int32_t cap = std::min(rank_cap, std::min(m, n));
      L.cap[b] = cap;
      L.slot[b] = L.n_slots++;
      L.x_off[b] = alloc((int64_t)m * cap);
      L.y_off[b] = alloc((int64_t)n * cap);
      fe += (int64_t)(m + n) * cap;
    }
  }
  L.factor_elems = fe;
  L.nrhs_max = nrhs_max;
  L.nrhs_slot = L.n_slots++;
  L.work_off = alloc((int64_t)C[0].size * nrhs_max);
  L.out_off = alloc((int64_t)C[0].size * nrhs_max);
  const int64_t ring =
      ring_elems > 0 ? ring_elems : std::min<int64_t>(std::max<int64_t>(8 * fe, int64_t(1) << 22), int64_t(1) << 31);
  L.ring_off = alloc(ring);
  L.ring_size = ring;
  const int32_t segsz = std::max(leafmax, tile);
  start = Schedule();
  iter = Schedule();
  apply = Schedule();
  std::vector<int32_t> dbuf, xbuf, ybuf;
  const int32_t A0 = 0, X0 = nb, T0 = 2 * nb, Y0 = 3 * nb;
  {
    Sched s(C, Bx, rank_cap, L, &start, dbuf, xbuf, ybuf, true, segsz, false, L.ring_off, ring);
    s.copy_scaled(X0, A0, 1.0f, true);
  }
  // (n = 6, FP64, eps 1e-8, twenty steps: 1.7 s accumulated, 8.1 s not)
  with_ring(tile > 0, L, [&](bool acc) {
    iter = Schedule();
    Sched s(C, Bx, rank_cap, L, &iter, dbuf, xbuf, ybuf, true, segsz, acc, L.ring_off, ring);
    s.zero(T0);
    s.gemm(T0, A0, X0, -1.0f);  // T = -A X
    s.settle_all(T0);
    s.copy_scaled(Y0, X0, 2.0f, false);
    s.gemm(Y0, X0, T0, 1.0f);   // Y = 2 X - X A X
    s.settle_all(Y0);
    s.copy_scaled(X0, Y0, 1.0f, false);
    st.temp_elems = s.temp_elems_;
    st.ring_wraps = s.wraps_;
    st.early_pieces = s.early_pieces_;
    st.accumulated = acc;
  });
  {
    Sched s(C, Bx, rank_cap, L, &apply, dbuf, xbuf, ybuf, true, segsz, false, L.ring_off, ring);
    const int32_t N = C[0].size;
    MV Win, Wout;
    Win.buf = -1;  // read-only here
    Win.clus = 0;
    Win.v = View{L.work_off, 1, N, N, nrhs_max, L.nrhs_slot, 0};
    Wout.buf = s.new_buf_leaves(0);
    Wout.clus = 0;
    Wout.v = View{L.out_off, 1, N, N, nrhs_max, L.nrhs_slot, 0};
    s.apply(X0, Win, Wout);
  }
  for (Schedule* sc : {&start, &iter, &apply}) sc->n_edges = (int64_t)sc->pred_idx.size();
  st.n_factor_tasks = (int64_t)iter.tasks.size();
  st.n_solve_tasks = (int64_t)apply.tasks.size();
  st.host_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
}

}  // namespace hlu
