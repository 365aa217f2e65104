// Mesh construction: validation of the leaf list, node enumeration, hanging-node detection and
// upload of the device tables (Sec. 5.2 "Octree construction and 2:1 balancing" and Sec. 5.3
// "Identification of unique, independent nodes").
//
// Instead of the paper's distributed sort of (element, node) edges, this builds flat index tables
// once on the host: every leaf emits its 8 corners (candidate nodes) and its 12 edge midpoints and
// 6 face centres ("cancellation" positions one level deeper). A corner that coincides with a
// cancellation position of some leaf lies inside that leaf's edge or face and is hanging; its
// parents are that edge's two ends (weight 1/2) or that face's four corners (weight 1/4), the
// interpolation from the immediate parent of Fig. "traversal". Under the full 2:1 balance the
// parents of a hanging node are never hanging themselves; this is checked.
#include <algorithm>
#include <array>
#include <atomic>
#include <cmath>
#include <cstring>
#include <iterator>
#include <memory>
#include <numeric>
#include <thread>

#include "internal.h"
#include "hostutil.h"

namespace chns {
namespace {

using host::compact3;
using host::kFull;
using host::morton;
using host::parallel_for;

// Corner c (0..7, bits x,y,z) of a leaf.
inline void corner_xyz(const uint32_t* a, uint64_t s, int c, uint64_t out[3]) {
  out[0] = a[0] + ((c & 1) ? s : 0);
  out[1] = a[1] + (((c >> 1) & 1) ? s : 0);
  out[2] = a[2] + (((c >> 2) & 1) ? s : 0);
}

// Cancellation position `kind` of a leaf and its parent corners (2 for edges, 4 for faces).
// Edges: kind = 4*d + (b1 + 2*b2): axis d, offsets b1,b2 on the two other axes (ascending).
// Faces: kind = 12 + 2*d + b: normal axis d at side b.
inline int cancel_geom(int kind, int par[4], int mid_half[3], int base_bits[3]) {
  if (kind < 12) {
    int d = kind / 4, r = kind % 4;
    int o1 = d == 0 ? 1 : 0, o2 = d == 2 ? 1 : 2;
    int b1 = r & 1, b2 = r >> 1;
    base_bits[0] = base_bits[1] = base_bits[2] = 0;
    base_bits[o1] = b1;
    base_bits[o2] = b2;
    mid_half[0] = mid_half[1] = mid_half[2] = 0;
    mid_half[d] = 1;
    int c0 = base_bits[0] | (base_bits[1] << 1) | (base_bits[2] << 2);
    par[0] = c0;
    par[1] = c0 | (1 << d);
    par[2] = par[3] = -1;
    return 2;
  }
  int f = kind - 12, d = f / 2, b = f % 2;
  int o1 = d == 0 ? 1 : 0, o2 = d == 2 ? 1 : 2;
  base_bits[0] = base_bits[1] = base_bits[2] = 0;
  base_bits[d] = b;
  mid_half[0] = mid_half[1] = mid_half[2] = 1;
  mid_half[d] = 0;
  int c0 = b << d;
  par[0] = c0;
  par[1] = c0 | (1 << o1);
  par[2] = c0 | (1 << o2);
  par[3] = c0 | (1 << o1) | (1 << o2);
  return 4;
}

}  // namespace

static chns_status alloc_workspace(chns_mesh* m, bool light) {
  const int64_t N = m->d.n_nodes;
  const size_t n3 = (size_t)(3 * N);
  Workspace& w = m->ws;
  if (light) {
    // level meshes of a multigrid hierarchy: operator applies and diagonals only (no Krylov
    // solve runs on them), so no solver vectors
    CHNS_CUDA(cudaStreamCreateWithFlags(&m->cap_stream, cudaStreamNonBlocking));
    return CHNS_OK;
  }
  // one allocation, cut into 256-byte aligned arrays (some forty cudaMalloc calls took longer than
  // the tables of a small mesh)
  w.v64.assign(kNumVec64, nullptr);
  w.v32.assign(kNumVec32, nullptr);
  struct Part {
    void** p;
    size_t bytes;
  };
  std::vector<Part> parts;
  auto part = [&](auto*& p, size_t count) {
    parts.push_back({(void**)&p, (count * sizeof(*p) + 255) / 256 * 256});
  };
  for (auto& p : w.v64) part(p, n3);
  for (auto& p : w.v32) part(p, n3);
  part(w.gm_V, (size_t)(CHNS_GMRES_MAX_RESTART + 1) * n3);
  part(w.gm_V32, (size_t)(CHNS_GMRES_MAX_RESTART + 1) * n3);
  part(w.red, (size_t)(kScalarBase + 1024));
  part(w.counter, 64);
  float* c32 = nullptr;
  __nv_bfloat16* c16 = nullptr;
  part(c32, (size_t)10 * N);
  part(c16, (size_t)8 * N);
  part(w.coef64, (size_t)16 * N);
  part(w.part_big, (size_t)(m->d.n_elem / 64 + 64));
  part(w.md_part, (size_t)(CHNS_GMRES_MAX_RESTART + 2) * kMdMaxBlocks);
  size_t total = 0;
  for (auto& q : parts) total += q.bytes;
  CHNS_CUDA(cudaMalloc(&w.slab, total));
  char* at = static_cast<char*>(w.slab);
  for (auto& q : parts) {
    *q.p = at;
    at += q.bytes;
  }
  w.coef32 = c32;
  w.coef16 = c16;
  CHNS_CUDA(cudaMemset(w.red, 0, (size_t)(kScalarBase + 1024) * sizeof(double)));
  CHNS_CUDA(cudaMemset(w.counter, 0, 64 * sizeof(unsigned int)));
  CHNS_CUDA(cudaMallocHost(&w.h_pinned, 1024 * sizeof(double)));
  CHNS_CUDA(cudaStreamCreateWithFlags(&m->cap_stream, cudaStreamNonBlocking));
  return CHNS_OK;
}

static void dfree(void* p) {
  if (p) cudaFree(p);
}

void free_mesh(chns_mesh* m) {
  if (!m) return;
  dfree(m->d_enode);
  dfree(m->d_level);
  dfree(m->d_hang);
  dfree(m->d_anchor);
  dfree(m->d_bnd);
  dfree(m->d_patch_elem);
  dfree(m->d_patch_head);
  dfree(m->d_rec);
  dfree(m->d_eloc);
  dfree(m->d_geo);
  dfree(m->d_node_int);
  Workspace& w = m->ws;
  dfree(w.slab);
  if (w.h_pinned) cudaFreeHost(w.h_pinned);
  dfree(m->mq.qd64);
  dfree(m->mq.qd32);
  for (int p = 0; p < 2; ++p)
    for (int k = 0; k < 2; ++k) dfree(m->sd.d[p][k]);
  dfree(m->qvu);
  if (m->cap_stream) cudaStreamDestroy(m->cap_stream);
  delete m;
}

// Greedy partition of the Morton-ordered elements into patches (see kPatchElems/kPatchSlots and
// the index record in internal.h): regular slots = distinct nodes used as corners or as parents
// of hanging corners, hanging slots = distinct hanging corners; a node is owned by a patch when no
// other patch has it as a slot. Bricks are never split, and the levels of a patch span at most
// kPatchLevelSpan. The leaf list is cut into chunks of kPatchChunk leaves (moved to the next unit) that
// are partitioned in parallel.
struct PatchTables {
  std::vector<int32_t> elem;  // per patch: first element
  std::vector<uint4> head;
  std::vector<uint32_t> rec;
  std::vector<uint4> eloc;
};

static_assert(kPatchSlots - 1 <= (int)kElocSlotMask && CHNS_MAXD - 1 <= (int)kElocLevelMask &&
                  kElocLevelShift + 5 <= 16,
              "patch slot and level must fit the first uint16 of eloc");

constexpr int64_t kPatchChunk = 32768;

namespace {

// Distinct keys of one patch with the slot each gets (open addressing, cleared by epoch).
class SlotMap {
 public:
  SlotMap() : key_(kSize), val_(kSize), epoch_(kSize, 0) {}
  void clear() { ++now_; }
  // position of the key; *fresh: it was not there
  int put(uint32_t k, bool* fresh) {
    uint32_t h = (k * 2654435761u) >> (32 - kBits);
    while (epoch_[h] == now_ && key_[h] != k) h = (h + 1) & (kSize - 1);
    *fresh = epoch_[h] != now_;
    if (*fresh) {
      epoch_[h] = now_;
      key_[h] = k;
    }
    return (int)h;
  }
  void erase_last(int pos) { epoch_[pos] = 0; }  // of the latest insertions, newest first
  int32_t& val(int pos) { return val_[pos]; }
  int32_t get(uint32_t k) {
    uint32_t h = (k * 2654435761u) >> (32 - kBits);
    while (epoch_[h] != now_ || key_[h] != k) h = (h + 1) & (kSize - 1);
    return val_[h];
  }

 private:
  static constexpr int kBits = 12, kSize = 1 << kBits;
  std::vector<uint32_t> key_;
  std::vector<int32_t> val_;
  std::vector<uint32_t> epoch_;
  uint32_t now_ = 0;
};

struct PatchBuilder {
  int64_t N;
  const std::vector<int32_t>& enode;
  const std::vector<int4>& hang;
  const uint8_t* levels;
  const std::vector<uint8_t>& unit;  // per leaf: 8 at the first leaf of a brick, else 1
  std::vector<uint4>& eloc;
  std::vector<int32_t> elem;
  std::vector<uint4> head;
  std::vector<uint32_t> rec;

  SlotMap map;
  std::vector<int32_t> reg, hg;  // ids of the current patch (node id with flags; hanging id)
  std::vector<int> fresh;

  int32_t slot_of(int32_t v) { return map.get((uint32_t)(v & kIdxMask)); }

  // adds the nodes of one unit; returns false (and takes them back) if the slots do not fit
  bool add_unit(int64_t e, int n, bool force) {
    const size_t r0 = reg.size(), h0 = hg.size();
    fresh.clear();
    auto node = [&](int32_t id) {
      bool f;
      const int pos = map.put((uint32_t)(id & kIdxMask), &f);
      if (f) {
        fresh.push_back(pos);
        reg.push_back(id);
      }
    };
    for (int64_t q = 8 * e; q < 8 * (e + n); ++q) {
      const int32_t v = enode[q], j = v & kIdxMask;
      if (j < N) {
        node(v);
        continue;
      }
      bool f;
      const int pos = map.put((uint32_t)j, &f);
      if (!f) continue;
      fresh.push_back(pos);
      const int32_t h = j - (int32_t)N;
      hg.push_back(h);
      const int4 p = hang[h];
      node(p.x);
      node(p.y);
      if (p.z >= 0) {
        node(p.z);
        node(p.w);
      }
    }
    if (force || reg.size() + hg.size() <= (size_t)kPatchSlots) return true;
    while (!fresh.empty()) {
      map.erase_last(fresh.back());
      fresh.pop_back();
    }
    reg.resize(r0);
    hg.resize(h0);
    return false;
  }

  void close(int64_t e0, int64_t e1, const std::vector<std::pair<int32_t, int32_t>>& units) {
    std::sort(reg.begin(), reg.end(),
              [](int32_t a, int32_t b) { return (a & kIdxMask) < (b & kIdxMask); });
    std::sort(hg.begin(), hg.end());
    const int nr = (int)reg.size(), nh = (int)hg.size();
    bool f;
    for (int i = 0; i < nr; ++i) map.val(map.put((uint32_t)(reg[i] & kIdxMask), &f)) = i;
    for (int i = 0; i < nh; ++i) map.val(map.put((uint32_t)(N + hg[i]), &f)) = nr + i;
    // corner slots of the elements
    std::vector<std::array<uint16_t, 8>> loc((size_t)(e1 - e0));
    for (int64_t e = e0; e < e1; ++e) {
      auto& l = loc[e - e0];
      for (int c = 0; c < 8; ++c) l[c] = (uint16_t)slot_of(enode[8 * e + c]);
      eloc[e] = make_uint4((l[0] | (uint32_t)levels[e] << kElocLevelShift) | (uint32_t)l[1] << 16,
                           l[2] | (uint32_t)l[3] << 16, l[4] | (uint32_t)l[5] << 16,
                           l[6] | (uint32_t)l[7] << 16);
    }
    std::vector<uint32_t> w;
    auto align = [&] { w.resize((w.size() + 3) / 4 * 4, 0); };
    for (int32_t id : reg) w.push_back((uint32_t)id);
    align();
    for (int i = 0; i < nh; ++i) {
      const int4 q = hang[hg[i]];
      const uint32_t ab = (uint32_t)slot_of(q.x) | (uint32_t)slot_of(q.y) << 16;
      w.push_back(ab);
      w.push_back(q.z < 0 ? ab : (uint32_t)slot_of(q.z) | (uint32_t)slot_of(q.w) << 16);
    }
    align();
    // references: brick pairs, then the other leaves two by two
    const uint32_t refs = (uint32_t)(w.size() / 4);
    int nb = 0, ns = 0, low = CHNS_MAXD;
    for (auto& u : units) {
      (u.second == 8 ? nb : ns) += 1;
      low = std::min(low, (int)levels[u.first]);
    }
    const int nb4 = 4 * nb, n2 = (ns + 1) / 2;
    std::vector<std::array<uint16_t, 16>> ref((size_t)(nb4 + n2));
    // level of leaf k of the patch in the upper bits of entry at
    auto tag = [&](std::array<uint16_t, 16>& r, int at, int k) {
      r[at] = (uint16_t)(r[at] | (uint32_t)(levels[e0 + k] - low) << 12);
    };
    int b = 0, s = 0;
    for (auto& u : units) {
      const int k0 = (int)(u.first - e0);
      if (u.second == 8) {
        for (int p = 0; p < 4; ++p) {
          const int lo = k0 + 2 * p;
          auto& r = ref[4 * b + p];
          for (int j = 0; j < 4; ++j)
            for (int ix = 0; ix < 3; ++ix)
              r[3 * j + ix] = (uint16_t)(4 * (ix < 2 ? loc[lo][ix + 2 * j] : loc[lo + 1][1 + 2 * j]));
          tag(r, 0, lo);
        }
        ++b;
      } else {
        auto& r = ref[nb4 + s / 2];
        for (int a = 0; a < 8; ++a) {
          r[8 * (s & 1) + a] = (uint16_t)(4 * loc[k0][a]);
          if (!(s & 1)) r[8 + a] = r[a];  // until there is a second leaf
        }
        tag(r, 8 * (s & 1), k0);
        if (s & 1) r[6] = (uint16_t)(r[6] | 1u << 12);
        ++s;
      }
    }
    auto put = [&](const std::array<uint16_t, 16>& r, int from, int halves) {
      for (int k = from; k < from + halves; k += 2)
        w.push_back((uint32_t)r[k] | (uint32_t)r[k + 1] << 16);
    };
    for (int j = 0; j < 3; ++j)
      for (int t = 0; t < nb4; ++t) put(ref[t], 4 * j, 4);
    align();
    for (int j = 0; j < 2; ++j)
      for (int t = 0; t < n2; ++t) put(ref[nb4 + t], 8 * j, 8);
    align();
    elem.push_back((int32_t)e0);
    head.push_back(make_uint4((uint32_t)(rec.size() / 4), (uint32_t)nr | (uint32_t)nh << 16,
                              (uint32_t)nb | (uint32_t)ns << 16, (uint32_t)low | refs << 16));
    rec.insert(rec.end(), w.begin(), w.end());
    reg.clear();
    hg.clear();
    map.clear();
  }

  void run(int64_t b, int64_t e) {
    std::vector<std::pair<int32_t, int32_t>> units;
    map.clear();
    int64_t e0 = b;
    int low = CHNS_MAXD, high = 0;  // levels of the current patch
    for (int64_t i = b; i < e;) {
      const int n = unit[i], l = levels[i];
      if (i > e0 && (i - e0 + n > kPatchElems ||
                     std::max(high, l) - std::min(low, l) > kPatchLevelSpan ||
                     !add_unit(i, n, false))) {
        close(e0, i, units);
        units.clear();
        e0 = i;
        low = CHNS_MAXD;
        high = 0;
        continue;
      }
      if (i == e0) add_unit(i, n, true);
      low = std::min(low, l);
      high = std::max(high, l);
      units.push_back({(int32_t)i, n});
      i += n;
    }
    if (e0 < e) close(e0, e, units);
  }
};

}  // namespace

static void build_patches(int64_t n, int64_t N, const uint32_t* anchors,
                          const std::vector<int32_t>& enode, const std::vector<int4>& hang,
                          const uint8_t* levels, PatchTables& P) {
  // bricks: 8 consecutive leaves of one level, the first at its parent's anchor
  std::vector<uint8_t> unit((size_t)n, 1);
  for (int64_t e = 0; e + 8 <= n;) {
    const int l = levels[e];
    bool brick = l > 0;
    const uint32_t sp = l > 0 ? (uint32_t)(kFull >> (l - 1)) : 1;
    for (int d = 0; d < 3 && brick; ++d) brick = anchors[3 * e + d] % sp == 0;
    for (int k = 1; k < 8 && brick; ++k) brick = levels[e + k] == l;
    if (brick) unit[e] = 8;
    e += brick ? 8 : 1;
  }
  std::vector<int64_t> cut{0};
  for (int64_t c = kPatchChunk; c < n; c += kPatchChunk) {
    int64_t e = c;  // not inside a brick
    for (int k = 1; k < 8; ++k)
      if (unit[c - k] == 8) e = c - k + 8;
    if (e < n && e > cut.back()) cut.push_back(e);
  }
  cut.push_back(n);
  P.eloc.resize(n);
  const int nc = (int)cut.size() - 1;
  std::vector<std::unique_ptr<PatchBuilder>> part(nc);
  std::atomic<int> next(0);
  const int nt = std::min(nc, (int)std::max(1u, std::min(16u, std::thread::hardware_concurrency())));
  host::parallel_parts(nt, nt, [&](int, int64_t, int64_t) {
    for (int c; (c = next.fetch_add(1)) < nc;) {
      part[c].reset(new PatchBuilder{N, enode, hang, levels, unit, P.eloc});
      part[c]->run(cut[c], cut[c + 1]);
    }
  });
  // concatenate; a node is owned by the only patch that has it as a regular slot
  std::vector<uint8_t> count((size_t)N, 0);
  for (auto& p : part) {
    const uint32_t base = (uint32_t)(P.rec.size() / 4);
    for (size_t k = 0; k < p->head.size(); ++k) {
      uint4 h = p->head[k];
      const uint32_t* r = &p->rec[4 * (size_t)h.x];
      h.x += base;
      P.elem.push_back(p->elem[k]);
      P.head.push_back(h);
      for (uint32_t i = 0; i < (h.y & 0xffffu); ++i) {
        uint8_t& c = count[r[i] & kNodeMask];
        c = (uint8_t)std::min(2, c + 1);
      }
    }
    P.rec.insert(P.rec.end(), p->rec.begin(), p->rec.end());
    p.reset();
  }
  P.elem.push_back((int32_t)n);
  parallel_for((int64_t)P.head.size(), [&](int64_t b, int64_t e) {
    for (int64_t k = b; k < e; ++k) {
      uint32_t* r = &P.rec[4 * (size_t)P.head[k].x];
      for (uint32_t i = 0; i < (P.head[k].y & 0xffffu); ++i)
        if (count[r[i] & kNodeMask] == 1) r[i] |= (uint32_t)kOwnBit;
    }
  });
}

chns_status build_mesh(const uint32_t* anchors, const uint8_t* levels, int64_t n,
                       const double extent[3], cudaStream_t stream, chns_mesh* m, bool light,
                       bool keep_host) {
  CHNS_CHECK(n > 0 && n < (int64_t(1) << 28), CHNS_EINVAL, "n_leaves out of range");
  for (int d = 0; d < 3; ++d)
    CHNS_CHECK(extent[d] > 0.0, CHNS_EINVAL, "extent must be positive");

  // ---- per-leaf checks: level range, alignment, Morton order, disjointness, coverage
  std::vector<uint64_t> lkey(n);
  int minl = CHNS_MAXD, maxl = 0;
  for (int64_t i = 0; i < n; ++i) {
    int l = levels[i];
    CHNS_CHECK(l < CHNS_MAXD, CHNS_EINVAL, "leaf level must be < CHNS_MAXD");
    uint64_t s = kFull >> l;
    for (int d = 0; d < 3; ++d) {
      uint64_t a = anchors[3 * i + d];
      CHNS_CHECK(a % s == 0 && a + s <= kFull, CHNS_EINVAL, "anchor not aligned or outside the cube");
    }
    lkey[i] = morton(anchors[3 * i], anchors[3 * i + 1], anchors[3 * i + 2]);
    minl = std::min(minl, l);
    maxl = std::max(maxl, l);
  }
  unsigned __int128 vol = 0;
  for (int64_t i = 0; i < n; ++i) {
    uint64_t span = 1ull << (3 * (CHNS_MAXD - levels[i]));
    vol += span;
    if (i + 1 < n)
      CHNS_CHECK(lkey[i] + span <= lkey[i + 1], CHNS_EINVAL,
                 "leaves are not in strictly increasing Morton order or overlap");
  }
  CHNS_CHECK(vol == ((unsigned __int128)1 << (3 * CHNS_MAXD)), CHNS_EINVAL,
             "leaves do not cover the unit cube");

  // ---- 2:1 balance across faces, edges and corners: the same-size neighbour in each of the 26
  // directions must lie in a leaf at most one level coarser.
  std::atomic<bool> unbalanced(false);
  parallel_for(n, [&](int64_t b, int64_t e) {
    for (int64_t i = b; i < e && !unbalanced.load(); ++i) {
      int l = levels[i];
      int64_t s = int64_t(kFull >> l);
      for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
          for (int dx = -1; dx <= 1; ++dx) {
            if (!dx && !dy && !dz) continue;
            int64_t p[3] = {int64_t(anchors[3 * i]) + dx * s + s / 2,
                            int64_t(anchors[3 * i + 1]) + dy * s + s / 2,
                            int64_t(anchors[3 * i + 2]) + dz * s + s / 2};
            if (p[0] < 0 || p[1] < 0 || p[2] < 0 || p[0] >= int64_t(kFull) ||
                p[1] >= int64_t(kFull) || p[2] >= int64_t(kFull))
              continue;
            uint64_t k = morton(p[0], p[1], p[2]);
            int64_t j = int64_t(std::upper_bound(lkey.begin(), lkey.end(), k) - lkey.begin()) - 1;
            if (j < 0 || int(levels[j]) < l - 1) unbalanced.store(true);
          }
    }
  });
  CHNS_CHECK(!unbalanced.load(), CHNS_EUNBALANCED, "leaves are not 2:1 balanced");

  // ---- unique corner points: the leaves' anchors (distinct and sorted already) and the corners that
  // are no leaf's anchor (on upper domain faces, and where a coarser leaf lies beyond), which alone
  // are sorted
  std::vector<uint64_t> ckey((size_t)n * 8);
  std::vector<uint64_t> pts;
  {
    const int nt = host::threads_for(n);
    std::vector<std::vector<uint64_t>> extra(nt);
    host::parallel_parts(n, nt, [&](int t, int64_t b, int64_t e) {
      for (int64_t i = b; i < e; ++i) {
        uint64_t s = kFull >> levels[i];
        for (int c = 0; c < 8; ++c) {
          uint64_t q[3];
          corner_xyz(anchors + 3 * i, s, c, q);
          const uint64_t k = morton(q[0], q[1], q[2]);
          ckey[8 * i + c] = k;
          if (c == 0) continue;
          // the next leaves in Morton order hold most of the anchors
          bool found = false;
          for (int64_t j = i + 1; j < std::min(i + 8, n) && !found; ++j) found = lkey[j] == k;
          if (!found && !std::binary_search(lkey.begin(), lkey.end(), k)) extra[t].push_back(k);
        }
      }
      std::sort(extra[t].begin(), extra[t].end());
      extra[t].erase(std::unique(extra[t].begin(), extra[t].end()), extra[t].end());
    });
    std::vector<uint64_t> all;
    for (auto& v : extra) {
      std::vector<uint64_t> m;
      m.reserve(all.size() + v.size());
      std::set_union(all.begin(), all.end(), v.begin(), v.end(), std::back_inserter(m));
      all.swap(m);
    }
    pts.resize((size_t)n + all.size());
    std::merge(lkey.begin(), lkey.end(), all.begin(), all.end(), pts.begin());
  }
  const int64_t NP = (int64_t)pts.size();

  // ---- hanging detection: a corner point at a cancellation position of some leaf (18 leaf + kind;
  // several leaves may report a point, all with the same parents). Leaves of the finest level have
  // nothing inside their edges and faces.
  std::vector<std::atomic<int64_t>> hang_src((size_t)NP);
  parallel_for(NP, [&](int64_t b, int64_t e) {
    for (int64_t p = b; p < e; ++p) hang_src[p].store(-1, std::memory_order_relaxed);
  });
  parallel_for(n, [&](int64_t b, int64_t e) {
    for (int64_t i = b; i < e; ++i) {
      if (levels[i] == maxl) continue;
      uint64_t s = kFull >> levels[i], h = s / 2;
      for (int k = 0; k < 18; ++k) {
        int par[4], mh[3], bb[3];
        cancel_geom(k, par, mh, bb);
        uint64_t q[3];
        for (int d = 0; d < 3; ++d) q[d] = anchors[3 * i + d] + bb[d] * s + mh[d] * h;
        const uint64_t key = morton(q[0], q[1], q[2]);
        auto it = std::lower_bound(pts.begin(), pts.end(), key);
        if (it != pts.end() && *it == key)
          hang_src[it - pts.begin()].store(18 * i + k, std::memory_order_relaxed);
      }
    }
  });

  // ---- numbering: independent nodes in Morton order (pts is sorted by Morton key)
  std::vector<int64_t> pid(NP);
  int64_t N = 0, H = 0;
  for (int64_t p = 0; p < NP; ++p) pid[p] = hang_src[p].load(std::memory_order_relaxed) < 0 ? N++ : -(++H);
  CHNS_CHECK(N < (int64_t(1) << 29) && H < (int64_t(1) << 29), CHNS_EINVAL, "mesh too large");

  auto point_index = [&](uint64_t key) -> int64_t {
    auto it = std::lower_bound(pts.begin(), pts.end(), key);
    if (it == pts.end() || *it != key) return -1;
    return int64_t(it - pts.begin());
  };

  m->node_coords.resize((size_t)3 * N);
  m->node_bnd.resize((size_t)N);
  parallel_for(NP, [&](int64_t b0, int64_t e0) {
    for (int64_t p = b0; p < e0; ++p) {
      if (pid[p] < 0) continue;
      uint64_t x = compact3(pts[p]), y = compact3(pts[p] >> 1), z = compact3(pts[p] >> 2);
      int64_t j = pid[p];
      m->node_coords[3 * j] = (uint32_t)x;
      m->node_coords[3 * j + 1] = (uint32_t)y;
      m->node_coords[3 * j + 2] = (uint32_t)z;
      bool b = x == 0 || y == 0 || z == 0 || x == kFull || y == kFull || z == kFull;
      m->node_bnd[j] = b ? 1 : 0;
    }
  });
  int64_t nb = 0;
  for (uint8_t v : m->node_bnd) nb += v;
  auto flagged = [&](int64_t j) -> int32_t {
    return (int32_t)j | (m->node_bnd[j] ? kDirBit : 0);
  };

  // hanging table
  std::vector<int4> hang((size_t)std::max<int64_t>(H, 1));
  std::atomic<bool> bad(false);
  parallel_for(NP, [&](int64_t b, int64_t e) {
    for (int64_t p = b; p < e; ++p) {
      if (pid[p] >= 0) continue;
      int64_t h = -pid[p] - 1;
      const int64_t src = hang_src[p].load(std::memory_order_relaxed), leaf = src / 18;
      int par[4], mh[3], bb[3];
      int np = cancel_geom((int)(src % 18), par, mh, bb);
      uint64_t s = kFull >> levels[leaf];
      int32_t out[4] = {-1, -1, -1, -1};
      for (int k = 0; k < np; ++k) {
        uint64_t q[3];
        corner_xyz(anchors + 3 * leaf, s, par[k], q);
        int64_t pp = point_index(morton(q[0], q[1], q[2]));
        if (pp < 0 || pid[pp] < 0) {
          bad.store(true);
          break;
        }
        out[k] = flagged(pid[pp]);
      }
      hang[h] = make_int4(out[0], out[1], out[2], out[3]);
    }
  });
  CHNS_CHECK(!bad.load(), CHNS_EUNBALANCED, "hanging node whose parent is not an independent node");

  // element corner table
  std::vector<int32_t> enode((size_t)n * 8);
  parallel_for(n, [&](int64_t b, int64_t e) {
    for (int64_t i = b; i < e; ++i)
      for (int c = 0; c < 8; ++c) {
        int64_t p = point_index(ckey[8 * i + c]);
        int64_t id = pid[p];
        enode[8 * i + c] = id >= 0 ? flagged(id) : (int32_t)(N + (-id - 1));
      }
  });

  if (keep_host) {
    m->h_enode = enode;
    m->h_hang.assign(hang.begin(), hang.begin() + H);
  }

  // ---- patches (CTA-level gather / scatter)
  PatchTables P;
  build_patches(n, N, anchors, enode, hang, levels, P);

  // ---- upload
  m->d.n_elem = n;
  m->d.n_nodes = N;
  m->d.n_hang = H;
  for (int d = 0; d < 3; ++d) m->d.ext[d] = extent[d];
  m->min_level = minl;
  m->max_level = maxl;
  m->n_boundary = nb;
  CHNS_CUDA(cudaMalloc(&m->d_enode, (size_t)n * 8 * sizeof(int32_t)));
  CHNS_CUDA(cudaMalloc(&m->d_level, (size_t)n));
  CHNS_CUDA(cudaMalloc(&m->d_hang, hang.size() * sizeof(int4)));
  CHNS_CUDA(cudaMalloc(&m->d_anchor, (size_t)n * 3 * sizeof(uint32_t)));
  CHNS_CUDA(cudaMemcpyAsync(m->d_enode, enode.data(), (size_t)n * 8 * sizeof(int32_t),
                            cudaMemcpyHostToDevice, stream));
  CHNS_CUDA(cudaMemcpyAsync(m->d_level, levels, (size_t)n, cudaMemcpyHostToDevice, stream));
  CHNS_CUDA(cudaMemcpyAsync(m->d_hang, hang.data(), hang.size() * sizeof(int4),
                            cudaMemcpyHostToDevice, stream));
  CHNS_CUDA(cudaMemcpyAsync(m->d_anchor, anchors, (size_t)n * 3 * sizeof(uint32_t),
                            cudaMemcpyHostToDevice, stream));
  {
    std::vector<int32_t> bl;
    bl.reserve((size_t)nb);
    for (int64_t j = 0; j < N; ++j)
      if (m->node_bnd[j]) bl.push_back((int32_t)j);
    CHNS_CUDA(cudaMalloc(&m->d_bnd, std::max<size_t>(bl.size(), 1) * sizeof(int32_t)));
    if (!bl.empty())
      CHNS_CUDA(cudaMemcpyAsync(m->d_bnd, bl.data(), bl.size() * sizeof(int32_t),
                                cudaMemcpyHostToDevice, stream));
    CHNS_CUDA(cudaStreamSynchronize(stream));
  }
  {
    const int64_t np = (int64_t)P.head.size();
    m->d.n_patch = np;
    CHNS_CUDA(cudaMalloc(&m->d_patch_elem, (np + 1) * sizeof(int32_t)));
    CHNS_CUDA(cudaMalloc(&m->d_patch_head, np * sizeof(uint4)));
    CHNS_CUDA(cudaMalloc(&m->d_rec, P.rec.size() * sizeof(uint32_t)));
    CHNS_CUDA(cudaMalloc(&m->d_eloc, (size_t)n * sizeof(uint4)));
    CHNS_CUDA(cudaMemcpy(m->d_patch_elem, P.elem.data(), (np + 1) * sizeof(int32_t), cudaMemcpyHostToDevice));
    CHNS_CUDA(cudaMemcpy(m->d_patch_head, P.head.data(), np * sizeof(uint4), cudaMemcpyHostToDevice));
    CHNS_CUDA(cudaMemcpy(m->d_rec, P.rec.data(), P.rec.size() * sizeof(uint32_t), cudaMemcpyHostToDevice));
    CHNS_CUDA(cudaMemcpy(m->d_eloc, P.eloc.data(), (size_t)n * sizeof(uint4), cudaMemcpyHostToDevice));
    m->d.patch_elem = m->d_patch_elem;
    m->d.patch_head = m->d_patch_head;
    m->d.rec = m->d_rec;
    m->d.eloc = m->d_eloc;
  }
  {
    std::vector<LevelGeo> geo(CHNS_MAXD);
    for (int l = 0; l < CHNS_MAXD; ++l) {
      const double sc = std::ldexp(1.0, -l);
      LevelGeo& G = geo[l];
      for (int d = 0; d < 3; ++d) {
        G.h[d] = extent[d] * sc;
        G.ih[d] = 1.0 / G.h[d];
        G.hf[d] = (float)G.h[d];
        G.ihf[d] = (float)G.ih[d];
      }
      G.detJ = G.h[0] * G.h[1] * G.h[2] * 0.125;
      G.detJf = (float)G.detJ;
    }
    CHNS_CUDA(cudaMalloc(&m->d_geo, CHNS_MAXD * sizeof(LevelGeo)));
    CHNS_CUDA(cudaMemcpy(m->d_geo, geo.data(), CHNS_MAXD * sizeof(LevelGeo), cudaMemcpyHostToDevice));
    m->d.geo = m->d_geo;
  }
  // node coordinates on the device (grid transfer of the learned preconditioner)
  CHNS_CUDA(cudaMalloc(&m->d_node_int, std::max<size_t>(m->node_coords.size(), 3) * sizeof(uint32_t)));
  CHNS_CUDA(cudaMemcpy(m->d_node_int, m->node_coords.data(),
                       m->node_coords.size() * sizeof(uint32_t), cudaMemcpyHostToDevice));
  m->d.enode = m->d_enode;
  m->d.level = m->d_level;
  m->d.hang = m->d_hang;
  m->d.anchor = m->d_anchor;
  int dev = 0;
  CHNS_CUDA(cudaGetDevice(&dev));
  m->device = dev;
  CHNS_CUDA(cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, dev));
  chns_status st = alloc_workspace(m, light);
  if (st != CHNS_OK) return st;
  CHNS_CUDA(cudaStreamSynchronize(stream));
  return CHNS_OK;
}

}  // namespace chns

extern "C" chns_status chns_mesh_create(const uint32_t* anchors, const uint8_t* levels,
                                        int64_t n_leaves, const double extent[3], void* stream,
                                        chns_mesh** out) {
  if (!anchors || !levels || !extent || !out) {
    chns::set_error("chns_mesh_create: null argument");
    return CHNS_EINVAL;
  }
  *out = nullptr;
  chns_mesh* m = new (std::nothrow) chns_mesh();
  if (!m) {
    chns::set_error("chns_mesh_create: out of host memory");
    return CHNS_ENOMEM;
  }
  chns_status st;
  try {
    st = chns::build_mesh(anchors, levels, n_leaves, extent, chns::as_stream(stream), m, false,
                          false);
  } catch (const std::bad_alloc&) {
    chns::set_error("chns_mesh_create: out of host memory");
    st = CHNS_ENOMEM;
  }
  if (st != CHNS_OK) {
    chns::free_mesh(m);
    return st;
  }
  *out = m;
  return CHNS_OK;
}

extern "C" chns_status chns_mesh_get_info(const chns_mesh* m, chns_mesh_info* info) {
  if (!m || !info) {
    chns::set_error("chns_mesh_get_info: null argument");
    return CHNS_EINVAL;
  }
  info->n_elem = m->d.n_elem;
  info->n_nodes = m->d.n_nodes;
  info->n_hanging = m->d.n_hang;
  info->n_boundary = m->n_boundary;
  info->min_level = m->min_level;
  info->max_level = m->max_level;
  for (int d = 0; d < 3; ++d) info->extent[d] = m->d.ext[d];
  return CHNS_OK;
}

extern "C" chns_status chns_mesh_set_apply_config(chns_mesh* m, chns_apply_kernel kernel,
                                                  int64_t max_ctas) {
  if (!m || max_ctas < 0 || (kernel != CHNS_APPLY_AUTO && kernel != CHNS_APPLY_PATCH &&
                             kernel != CHNS_APPLY_STREAM)) {
    chns::set_error("chns_mesh_set_apply_config: null mesh, unknown kernel or max_ctas < 0");
    return CHNS_EINVAL;
  }
  m->apply_kernel = kernel;
  m->apply_max_ctas = max_ctas;
  return CHNS_OK;
}

extern "C" chns_status chns_mesh_node_coords(const chns_mesh* m, uint32_t* coords) {
  if (!m || !coords) {
    chns::set_error("chns_mesh_node_coords: null argument");
    return CHNS_EINVAL;
  }
  std::memcpy(coords, m->node_coords.data(), m->node_coords.size() * sizeof(uint32_t));
  return CHNS_OK;
}

extern "C" chns_status chns_mesh_boundary(const chns_mesh* m, uint8_t* flags) {
  if (!m || !flags) {
    chns::set_error("chns_mesh_boundary: null argument");
    return CHNS_EINVAL;
  }
  std::memcpy(flags, m->node_bnd.data(), m->node_bnd.size());
  return CHNS_OK;
}

extern "C" void chns_mesh_destroy(chns_mesh* m) { chns::free_mesh(m); }
