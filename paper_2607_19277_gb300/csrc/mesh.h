// Host book-keeping of the block octree (paper Section 2.1.2 and Figs. 1-2: the grid,
// its connectivity and the refine/coarsen decisions live on the host; data stays on the
// device). Leaves are kept sorted by level, then Morton index.
#pragma once
#include <stdint.h>

#include <string>
#include <vector>

#include "agile_internal.h"

namespace agile {

struct Key {
  int lev, x, y, z;
};

inline uint64_t key_code(const Key& k) {
  return ((uint64_t)k.lev << 57) | ((uint64_t)(uint32_t)k.x << 38) |
         ((uint64_t)(uint32_t)k.y << 19) | (uint64_t)(uint32_t)k.z;
}

uint64_t morton3(uint32_t x, uint32_t y, uint32_t z);

// Open-addressing table from key codes (never 0: levels start at 1) to integers, in two flat
// arrays at most half full: a regrid builds and asks such tables tens of thousands of times.
class KeyTable {
 public:
  explicit KeyTable(size_t n = 0) { reset(n); }
  void reset(size_t n) {             // empty, with room for n keys
    size_t cap = 64;
    shift_ = 64 - 6;
    while (cap < 2 * n) {
      cap *= 2;
      --shift_;
    }
    keys_.assign(cap, 0);
    vals_.assign(cap, 0);
    size_ = 0;
  }
  bool insert(uint64_t code, int val = 0) {   // false when the key is there already
    if (2 * (size_ + 1) > keys_.size()) grow();
    const size_t i = slot(code);
    if (keys_[i]) return false;
    keys_[i] = code;
    vals_[i] = val;
    ++size_;
    return true;
  }
  int find(uint64_t code) const {    // its value, -1 without the key
    const size_t i = slot(code);
    return keys_[i] ? vals_[i] : -1;
  }

 private:
  size_t slot(uint64_t code) const {  // where the key is or would be
    const size_t mask = keys_.size() - 1;
    size_t i = (size_t)((code * 0x9E3779B97F4A7C15ull) >> shift_);   // the product's high bits
    while (keys_[i] && keys_[i] != code) i = (i + 1) & mask;
    return i;
  }
  void grow() {
    std::vector<uint64_t> k;
    std::vector<int> v;
    k.swap(keys_);
    v.swap(vals_);
    reset(k.size());
    for (size_t i = 0; i < k.size(); ++i)
      if (k[i]) insert(k[i], v[i]);
  }
  std::vector<uint64_t> keys_;
  std::vector<int> vals_;
  size_t size_ = 0;
  int shift_ = 0;
};

struct FaceInfo {
  int kind;      // FK_*
  int bc;        // BC_* for FK_BC
  int nbr[4];    // same: [0]; coarser: [0]; finer: t1 + 2 t2
  int par[3];    // coarser: neighbour block position parity
};

struct RegridPlan {
  std::vector<Key> blocks;         // new leaves in order
  std::vector<RegridSrc> src;      // per new leaf
  std::vector<int> created;        // indices (new order) of refined children / new parents
  int n_refined = 0;
  int n_coarsened = 0;
};

class HostMesh {
 public:
  HostMesh(const int base[3], int max_level, const int bc[6], const double xmin[3],
           const double xmax[3]);

  const std::vector<Key>& blocks() const { return blocks_; }
  int find(const Key& k) const;
  bool has(const Key& k) const { return find(k) >= 0; }
  int nblocks_dim(int lev, int d) const { return base_[d] << (lev - 1); }
  double dx(int lev, int d) const;
  // Block position moved by (dx, dy, dz) at its level, wrapped on periodic axes;
  // false when it leaves the domain.
  bool neighbour_pos(const Key& k, int ox, int oy, int oz, Key* out) const;
  FaceInfo face(int i, int f) const;
  // Leaf covering block position k (level k.lev or coarser), -1 if k is refined.
  int covering_leaf(const Key& k) const;

  RegridPlan plan(const std::vector<int>& flags) const;   // flags per leaf: +1/-1/0
  void apply(const RegridPlan& p);

  // Device descriptors for the current mesh.
  void build_descs(std::vector<BlockDesc>* desc, std::vector<GhostTask>* ghosts,
                   std::vector<FixupTask>* fixups, int* nslots, std::string* err) const;

  bool balanced() const;

 private:
  void reindex();
  int base_[3];
  int max_level_;
  int bc_[6];
  bool periodic_[3];
  double xmin_[3], xmax_[3];
  std::vector<Key> blocks_;
  KeyTable index_;
};

}  // namespace agile
