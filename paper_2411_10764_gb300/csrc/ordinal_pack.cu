// Builds the ordinal form of a model on the host (layout: ordinal.cuh).  Host
// code only.  Every load of a V or P model pays for it: 600 trees of depth 10
// over 96 features take 3.3 ms on 8 threads, 2,000 of depth 12 over 256 features
// 29 ms (aarch64).
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstring>
#include <limits>
#include <memory>
#include <thread>
#include <vector>

#include "mlt.h"
#include <cuda_fp16.h>

#include "ordinal.cuh"

namespace mlt {
namespace {

// Bytes of thresholds and lookup tables that a feature group aims at (every CTA
// of the ordinal kernel copies its group's).
constexpr uint32_t kGroupBytes = 120 * 1024;
constexpr uint32_t kGroupMaxBytes = 220 * 1024;  // more thresholds in eight features: no ordinal form

// A threshold's place in the order of the floats (+0 counts as -0).
uint32_t order_key(float v) {
  uint32_t u;
  if (v == 0.0f) v = -0.0f;
  std::memcpy(&u, &v, 4);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
float order_value(uint32_t k) {
  const uint32_t u = (k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k;
  float v;
  std::memcpy(&v, &u, 4);
  return v;
}
uint32_t bits_of(float v) {
  uint32_t u;
  std::memcpy(&u, &v, 4);
  return u;
}

// Lookup table over one feature's thresholds (ascending): the kernel's bucket
// of a value, the number of buckets and the thresholds of the fullest one.
struct Buckets {
  float lo = 0.0f, add = 0.0f;
  uint32_t base = 0, shift = 0, count = 1, most = 0;
  uint32_t at(float t) const { return (bits_of((t > lo ? t : lo) + add) - base) >> shift; }
};
// Steps of a search among m thresholds.
uint32_t steps_for(uint32_t m) {
  uint32_t s = 0;
  while ((1u << s) <= m) ++s;
  return s;
}
// Thresholds of the fullest bucket, bucket ids (ascending) shifted right by
// `shift`; looked no further once there are `enough`.
uint32_t fullest(const std::vector<uint32_t>& ids, uint32_t shift, uint32_t enough) {
  uint32_t most = 0, run = 0, last = 0xFFFFFFFFu;
  for (uint32_t id : ids) {
    const uint32_t at = id >> shift;
    run = at == last ? run + 1 : 1;
    last = at;
    if (run > most && (most = run) >= enough) break;
  }
  return most;
}
// The lookup table of ascending thresholds t: over the offsets c, the most
// buckets allowed that leave the fewest steps; then the fewest buckets that
// leave as few.  `ids` is working memory.
Buckets choose_buckets(const std::vector<float>& t, std::vector<uint32_t>& ids) {
  const double range = std::min(3.0e38, std::max(1e-30, static_cast<double>(t.back()) - t.front()));
  const size_t m = t.size();
  ids.resize(m);
  Buckets best;
  for (int q = 0; q < 26; q += 2) {
    const float c = std::max(1e-30f, static_cast<float>(std::ldexp(range, 1 - q)));
    Buckets b;
    b.lo = t.front();
    b.add = c - b.lo;
    b.base = bits_of(b.lo + b.add);
    while (b.at(t.back()) >= static_cast<uint32_t>(kOrdMaxBuckets)) ++b.shift;
    for (size_t i = 0; i < m; ++i) ids[i] = b.at(t[i]);
    // fewer steps than the best offset's: fewer than half of 2^steps thresholds
    const uint32_t enough = q == 0 ? 0xFFFFFFFFu : (1u << steps_for(best.most)) / 2;
    b.most = fullest(ids, 0, enough);
    if (q == 0 || b.most < enough) best = b;
  }
  best.count = best.at(t.back()) + 1;
  for (size_t i = 0; i < m; ++i) ids[i] = best.at(t[i]);
  uint32_t shift = 0;
  const uint32_t enough = 1u << steps_for(best.most);
  while ((ids[m - 1] >> shift) > 0 && fullest(ids, shift + 1, enough) < enough) ++shift;
  best.shift += shift;
  best.count = (ids[m - 1] >> shift) + 1;
  return best;
}

// Ascending order of the high words (a radix sort by 11 bits at a time; a
// comparison sort of the 6,400 splits of a feature took six times as long).
void sort_by_key(uint64_t* v, size_t n, std::vector<uint64_t>& other) {
  if (n < 512) {
    std::sort(v, v + n);
    return;
  }
  other.resize(n);
  uint64_t *from = v, *to = other.data();
  uint32_t at[3][2048] = {};
  for (size_t i = 0; i < n; ++i)
    for (int d = 0; d < 3; ++d) ++at[d][(v[i] >> (32 + 11 * d)) & 2047u];
  for (int d = 0; d < 3; ++d) {
    uint32_t sum = 0;
    for (uint32_t& a : at[d]) {
      const uint32_t count = a;
      a = sum;
      sum += count;
    }
    for (size_t i = 0; i < n; ++i) to[at[d][(from[i] >> (32 + 11 * d)) & 2047u]++] = from[i];
    std::swap(from, to);
  }
  std::memcpy(v, from, n * sizeof(uint64_t));  // three passes end in `other`
}

// Threads for n items that hold `nodes` nodes in all.  Below 4,096 nodes a
// thread the start of the threads shows: a V and a P model of 50 and 100 trees of
// depth 6 loaded in 1.3 ms with eight, 0.7 ms with this rule (aarch64 host, 16
// cores).
int worker_count(int n, size_t nodes) {
  const size_t most = std::min<size_t>(std::min(8u, std::thread::hardware_concurrency()), nodes / 4096);
  return std::max(1, std::min<int>(static_cast<int>(most), n / 8));
}

// Threads that share the steps of one packing.  run(n, body) calls body(i, w)
// for i in [0, n), item i on worker i % workers(), and returns false if one could
// not finish: no exception leaves a thread, and a thread that cannot be had is
// done without.  Started once, for starting seven takes 0.2 ms and there are five
// steps; between them the threads yield, later sleep.
class Crew {
 public:
  explicit Crew(int workers) {
    try {
      threads_.reserve(workers);
      while (static_cast<int>(threads_.size()) + 1 < workers)
        threads_.emplace_back([this, w = static_cast<int>(threads_.size()) + 1] { serve(w); });
    } catch (...) {
    }
    workers_ = static_cast<int>(threads_.size()) + 1;
  }
  ~Crew() {
    job_ = nullptr;
    step_.fetch_add(1, std::memory_order_release);
    for (std::thread& t : threads_) t.join();
  }
  int workers() const { return workers_; }
  template <typename F>
  bool run(int n, F&& body) {
    struct Job {
      F& body;
      int n, workers;
      std::atomic<bool> ok{true};
    } job{body, n, workers_};
    arg_ = &job;
    job_ = [](void* p, int w) {
      Job& j = *static_cast<Job*>(p);
      try {
        for (int i = w; i < j.n; i += j.workers) j.body(i, w);
      } catch (...) {
        j.ok = false;
      }
    };
    busy_.store(static_cast<int>(threads_.size()), std::memory_order_relaxed);
    step_.fetch_add(1, std::memory_order_release);
    job_(arg_, 0);
    while (busy_.load(std::memory_order_acquire) > 0) std::this_thread::yield();
    return job.ok;
  }

 private:
  void serve(int w) {
    for (unsigned seen = 0;; ++seen) {
      for (int tries = 0; step_.load(std::memory_order_acquire) == seen; ++tries) {
        if (tries < 1000)
          std::this_thread::yield();
        else
          std::this_thread::sleep_for(std::chrono::microseconds(20));
      }
      if (job_ == nullptr) return;
      job_(arg_, w);
      busy_.fetch_sub(1, std::memory_order_release);
    }
  }
  std::vector<std::thread> threads_;
  int workers_ = 1;
  void (*job_)(void*, int) = nullptr;
  void* arg_ = nullptr;
  std::atomic<unsigned> step_{0};
  std::atomic<int> busy_{0};
};

bool pack(const mlt_node* nodes, int n_trees, int depth, int F, bool round_half, std::vector<unsigned char>& out,
          OrdTable& t) {
  const int slots = (2 << depth) - 1;
  const size_t total_nodes = static_cast<size_t>(n_trees) * slots;
  const bool deep = depth > kMaxFullDepth;
  const int padded = (n_trees + kOrdTreePad - 1) / kOrdTreePad * kOrdTreePad;
  if (deep && F > kOrdDeepMaxF) return false;
  const uint32_t tree_words = (deep ? ord_head_bytes(kOrdHead) : ord_tree_bytes(depth)) / 4;
  auto value = [&](const mlt_node& nd) {
    return round_half ? __half2float(__float2half_rn(nd.value)) : nd.value;
  };
  // the most that the lookup tables and what describes them can take (checked
  // below), so that `out` is allocated once
  const int F8 = (F + 7) / 8 * 8;
  const size_t other_bytes = static_cast<size_t>(F8 / 8) * (kGroupMaxBytes + sizeof(OrdGroup)) + F8 * sizeof(OrdFeature) + 512;
  const size_t tail_word = static_cast<size_t>(padded) * tree_words;  // a deep model's blocks follow the heads
  if (tail_word >= 0x7FFFFFFFull) return false;
  std::vector<uint32_t> heads;  // deep: until the tail's size is known
  if (deep) {
    heads.resize(tail_word, 0u);
  } else {
    out.reserve(tail_word * 4 + other_bytes);
    out.resize(tail_word * 4, 0);
  }
  uint32_t* words = deep ? heads.data() : reinterpret_cast<uint32_t*>(out.data());

  // the tables with every word but the ordinals, and the split nodes as
  // (feature, threshold's order key, word index), on a few threads that take
  // consecutive trees; a deep model's blocks are numbered within a thread's share
  // until all are counted
  struct Split {
    uint32_t feature;
    uint32_t key;
    uint32_t word;
  };
  struct Root {
    uint32_t block;
    int node;
  };
  struct alignas(128) Worker {  // no two on one cache line
    std::vector<Split> splits;
    std::vector<uint32_t> per_feature;
    std::vector<unsigned char> reach;
    std::vector<float> inherit;
    std::vector<Root> queue;
    std::vector<uint32_t> blocks;  // deep: the tail
    size_t first_block = 0;        // of this share in the whole tail
    std::vector<uint64_t> other;   // working memory of the features' step
    std::vector<uint32_t> ids;
    std::vector<size_t> at;        // where this share's next split of a feature goes
    int first = 0, last = 0;       // its trees
    bool usable = true;
    double visits = 0.0;
  };
  std::vector<float> reached(slots);  // share of the candidates that a random path brings to a slot
  for (int j = 0; j < slots; ++j) reached[j] = j == 0 ? 1.0f : 0.5f * reached[(j - 1) / 2];
  const int levels = deep ? kOrdHead : depth;  // of the complete heap
  const int inner = (1 << levels) - 1;
  auto put_split = [&](Worker& k, const mlt_node& nd, int j, size_t word, uint32_t* at) {
    const float v = value(nd);
    k.usable = k.usable && v != -INFINITY;  // every number is >= it: no ordinal stands for that
    k.splits.push_back({static_cast<uint32_t>(nd.feature), order_key(v), static_cast<uint32_t>(word)});
    ++k.per_feature[nd.feature];
    *at = ord_offset(nd.feature) | (nd.default_left ? (deep ? kOrdNan : 1u) : 0u);
    k.visits += reached[j];
  };
  auto put_tree = [&](Worker& k, int tr) {
    std::vector<unsigned char>& reach = k.reach;
    std::vector<float>& inherit = k.inherit;
    std::vector<Root>& queue = k.queue;
    std::vector<uint32_t>& blocks = k.blocks;
    const mlt_node* nd = nodes + static_cast<size_t>(tr) * slots;
    const size_t base = static_cast<size_t>(tr) * tree_words;
    std::fill(reach.begin(), reach.end(), 0);
    reach[0] = 1;
    for (int j = 0; j < slots; ++j)
      if (reach[j] && nd[j].feature >= 0) reach[2 * j + 1] = reach[2 * j + 2] = 1;
    queue.clear();
    auto new_blocks = [&](uint32_t count) {
      const uint32_t first = static_cast<uint32_t>(blocks.size() / 8);
      blocks.resize(blocks.size() + 8 * count, 0u);
      return first;
    };
    for (int j = 0; j < 2 * inner + 1; ++j) {
      const bool split = reach[j] && nd[j].feature >= 0;
      inherit[j] = !reach[j] ? inherit[(j - 1) / 2] : split ? 0.0f : value(nd[j]);
      if (j < inner) {
        if (split) put_split(k, nd[j], j, base + j + 1, &words[base + j + 1]);
        continue;
      }
      // the leaves below each path (full), or the exits (deep)
      const size_t w = deep ? base + (1u << levels) + 2 * (j - inner) : base + j + 1;
      if (!split) {
        std::memcpy(&words[w], &inherit[j], 4);
        if (deep) words[w + 1] = kOrdExitLeaf;
        continue;
      }
      put_split(k, nd[j], j, w, &words[w]);
      const uint32_t first = new_blocks(2);
      words[w + 1] = first;
      queue.push_back({first, 2 * j + 1});
      queue.push_back({first + 1, 2 * j + 2});
    }
    for (size_t q = 0; q < queue.size(); ++q) {
      const Root root = queue[q];
      const size_t at = static_cast<size_t>(root.block) * 8;
      int node[8];
      uint32_t leaves = 0;
      bool more = false;
      node[1] = root.node;
      for (int i = 1; i < 8; ++i) {
        if (i > 1) node[i] = node[i >> 1] < 0 ? -1 : 2 * node[i >> 1] + 1 + (i & 1);
        if (node[i] < 0 || node[i] >= slots || !reach[node[i]]) {
          node[i] = -1;
          continue;
        }
        const mlt_node& n = nd[node[i]];
        if (n.feature < 0) {
          const float v = value(n);
          std::memcpy(&blocks[at + i], &v, 4);
          leaves |= 1u << i;
        } else {
          uint32_t word;
          put_split(k, n, node[i], tail_word + at + i, &word);
          blocks[at + i] = word;
          more = more || i >= 4;
        }
      }
      uint32_t next = 0;
      if (more) {
        next = new_blocks(8);
        for (int i = 4; i < 8; ++i)
          if (node[i] >= 0 && nd[node[i]].feature >= 0)
            for (int side = 0; side < 2; ++side)
              queue.push_back({next + static_cast<uint32_t>(2 * (i - 4) + side), 2 * node[i] + 1 + side});
      }
      blocks[at] = next | (leaves >> 1) << kOrdBlockBits;
    }
    k.usable = k.usable && blocks.size() / 8 < (1u << kOrdBlockBits);
  };
  Crew crew(worker_count(n_trees, total_nodes));
  const int workers = crew.workers();
  std::vector<Worker> made(workers);
  const bool built = crew.run(workers, [&](int w, int) {
    Worker& k = made[w];
    k.per_feature.assign(F + 1, 0u);
    k.reach.resize(slots);
    k.inherit.resize(slots);
    k.first = static_cast<int>(static_cast<long long>(n_trees) * w / workers);
    k.last = static_cast<int>(static_cast<long long>(n_trees) * (w + 1) / workers);
    if (!deep) k.splits.reserve(static_cast<size_t>(k.last - k.first) * inner);
    for (int tr = k.first; tr < k.last && k.usable; ++tr) put_tree(k, tr);
  });
  if (!built) return false;
  double visits = 0.0;
  size_t n_blocks = 0;
  for (Worker& k : made) {
    if (!k.usable) return false;
    visits += k.visits;
    k.first_block = n_blocks;
    n_blocks += k.blocks.size() / 8;
  }
  if (n_blocks >= (1u << kOrdBlockBits) || tail_word + 8 * n_blocks >= 0x7FFFFFFFull) return false;
  if (deep)  // the padding trees' exits are leaves of +0
    for (int tr = n_trees; tr < padded; ++tr)
      for (uint32_t e = 0; e < (1u << levels); ++e)
        words[static_cast<size_t>(tr) * tree_words + (1u << levels) + 2 * e + 1] = kOrdExitLeaf;
  size_t n_words = tail_word;
  if (deep) {
    n_words += 8 * std::max<size_t>(n_blocks, 1);  // finished walkers read block 0
    out.reserve(n_words * 4 + other_bytes);
    out.resize(n_words * 4, 0);
    words = reinterpret_cast<uint32_t*>(out.data());
    std::memcpy(words, heads.data(), tail_word * 4);
    crew.run(workers, [&](int w, int) {  // no allocation in it: nothing to fail
      Worker& k = made[w];
      const uint32_t base = static_cast<uint32_t>(k.first_block), mask = (1u << kOrdBlockBits) - 1u;
      for (int tr = k.first; tr < k.last; ++tr)
        for (uint32_t e = 0; e < (1u << levels); ++e) {
          uint32_t& exit = words[static_cast<size_t>(tr) * tree_words + (1u << levels) + 2 * e + 1];
          if (exit != kOrdExitLeaf) exit += base;
        }
      for (size_t i = 0; i < k.blocks.size(); i += 8)
        if (k.blocks[i] & mask) k.blocks[i] += base;  // a root's children come after it, never at 0
      if (!k.blocks.empty())
        std::memcpy(&words[tail_word + 8 * k.first_block], k.blocks.data(), k.blocks.size() * 4);
      for (Split& s : k.splits)
        if (s.word >= tail_word) s.word += 8 * base;
    });
  }

  // thresholds of every feature in order, and each node's place among them
  std::vector<size_t> start(F + 1, 0);
  for (int f = 0; f < F; ++f) {
    start[f + 1] = start[f];
    for (const Worker& k : made) start[f + 1] += k.per_feature[f];
  }
  const std::unique_ptr<uint64_t[]> sorted(new uint64_t[start[F]]);  // written before it is read
  {
    std::vector<size_t> at(start.begin(), start.end() - 1);
    for (Worker& k : made) {
      k.at = at;
      for (int f = 0; f < F; ++f) at[f] += k.per_feature[f];
    }
  }
  crew.run(workers, [&](int w, int) {  // no allocation in it
    Worker& k = made[w];
    for (const Split& s : k.splits) sorted[k.at[s.feature]++] = (static_cast<uint64_t>(s.key) << 32) | s.word;
  });
  std::vector<std::vector<float>> keys(F);  // distinct thresholds, ascending
  std::vector<Buckets> buckets(F);
  std::vector<unsigned char> fits(F, 1);
  if (!crew.run(F, [&](int f, int w) {
    std::vector<uint64_t>& other = made[w].other;
    std::vector<uint32_t>& ids = made[w].ids;
    uint64_t *b = sorted.get() + start[f], *e = sorted.get() + start[f + 1];
    sort_by_key(b, static_cast<size_t>(e - b), other);
    std::vector<float>& k = keys[f];
    uint32_t before = 0;
    for (const uint64_t* it = b; it != e; ++it) {
      const uint32_t key = static_cast<uint32_t>(*it >> 32);
      if (k.empty() || before != key) k.push_back(order_value(key));
      before = key;
      if (k.size() > static_cast<size_t>(kOrdMaxDistinct)) {
        fits[f] = 0;
        return;
      }
      words[static_cast<uint32_t>(*it)] |= static_cast<uint32_t>(k.size() - 1) << 16;
    }
    if (!k.empty()) buckets[f] = choose_buckets(k, ids);
      }))
    return false;
  if (std::find(fits.begin(), fits.end(), 0) != fits.end()) return false;
  // the table is padded to a multiple of 8 features; one without thresholds
  // has a bucket of its own and nothing but padding (ordinal 0)
  keys.resize(F8);
  buckets.resize(F8);
  std::vector<OrdFeature> feat(F8, OrdFeature{});
  std::vector<OrdGroup> groups;
  uint32_t total = 0;
  t.max_bytes = 0;
  for (int f = 0; f < F8; f += 8) {
    // features 4 apart are searched together with the larger number of
    // compares; a search may read 2^steps - 1 entries past the bucket's start
    auto steps_of = [&](int q) {
      const int other = (q & 4) ? q - 4 : q + 4;  // f is a multiple of 8
      return std::max(steps_for(buckets[q].most), steps_for(buckets[other].most));
    };
    uint32_t most = 0;  // unaligned rows: all eight together
    for (int q = f; q < f + 8; ++q) most = std::max(most, steps_for(buckets[q].most));
    auto thr_bytes = [&](int q) { return static_cast<uint32_t>((keys[q].size() + (1u << most)) * 4 + 15) & ~15u; };
    auto lut_bytes = [&](int q) { return (buckets[q].count * 2u + 15u) & ~15u; };
    uint32_t eight = 0;
    for (int q = f; q < f + 8; ++q) eight += thr_bytes(q) + lut_bytes(q);
    if (eight > kGroupMaxBytes) return false;
    if (groups.empty() || groups.back().bytes + eight > kGroupBytes) {
      t.chunks[groups.size()] = 0;
      groups.push_back({static_cast<uint32_t>(f), 0u, total, 0u});
    }
    OrdGroup& g = groups.back();
    ++t.chunks[groups.size() - 1];
    g.count += static_cast<uint32_t>(std::min(8, F - f));
    for (int q = f; q < f + 8; ++q) {
      feat[q].thr = g.bytes;
      feat[q].lut = g.bytes + thr_bytes(q);
      feat[q].lo = buckets[q].lo;
      feat[q].add = buckets[q].add;
      feat[q].base = buckets[q].base;
      feat[q].shift = buckets[q].shift;
      feat[q].last = buckets[q].count - 1;
      feat[q].steps = steps_of(q) | most << 8;
      g.bytes += thr_bytes(q) + lut_bytes(q);
    }
    total += eight;
    t.max_bytes = std::max(t.max_bytes, g.bytes);
  }
  auto room = [&](size_t bytes) {  // in `out`, on a 128-byte boundary
    const size_t at = (out.size() + 127) & ~static_cast<size_t>(127);
    out.resize(at + bytes, 0);
    return at;
  };
  t.off_image = room(total);
  unsigned char* const image = out.data() + t.off_image;
  std::vector<uint32_t> image_at(F8);
  for (const OrdGroup& g : groups)
    for (uint32_t q = g.first; q < (g.first + g.count + 7) / 8 * 8; ++q) image_at[q] = g.off;
  const bool filled = crew.run(F8, [&](int q, int) {
    float* thr = reinterpret_cast<float*>(image + image_at[q] + feat[q].thr);
    uint16_t* lut = reinterpret_cast<uint16_t*>(image + image_at[q] + feat[q].lut);
    for (uint32_t i = 0; i < (feat[q].lut - feat[q].thr) / 4; ++i)
      thr[i] = i < keys[q].size() ? keys[q][i] : std::numeric_limits<float>::quiet_NaN();
    uint32_t b = 0;  // lut[b] = thresholds in the buckets below b
    for (uint32_t at = 0; at < keys[q].size(); ++at) {
      const uint32_t end = std::min(buckets[q].count, buckets[q].at(keys[q][at]) + 1);
      while (b < end) lut[b++] = static_cast<uint16_t>(at);
    }
    while (b < buckets[q].count) lut[b++] = static_cast<uint16_t>(keys[q].size());
  });
  if (!filled) return false;

  auto append = [&](const void* p, size_t bytes) {
    const size_t at = room(bytes);
    std::memcpy(out.data() + at, p, bytes);
    return at;
  };
  t.off_table = 0;
  t.off_tail = t.off_table + tail_word * 4;
  t.visits = deep ? static_cast<float>(visits) : static_cast<float>(n_trees) * depth;  // a full walk has no early end
  t.rounds = deep ? (depth - kOrdHead + 2) / 3 : 0;
  t.off_features = append(feat.data(), feat.size() * sizeof(OrdFeature));
  t.off_groups = append(groups.data(), groups.size() * sizeof(OrdGroup));
  t.n_trees = padded;
  t.n_groups = static_cast<int>(groups.size());
  t.round_half = round_half ? 1 : 0;
  return true;
}
}  // namespace

bool pack_ordinal(const mlt_node* nodes, int n_trees, int depth, int F, bool round_half,
                  std::vector<unsigned char>& out, OrdTable& t) {
  bool ok = false;
  out.clear();
  try {
    ok = pack(nodes, n_trees, depth, F, round_half, out, t);
  } catch (const std::exception&) {  // no memory: the model does without
  }
  if (!ok) {
    out.clear();
    t = OrdTable();
  }
  return ok;
}

}  // namespace mlt
