// tiles.cpp -- tiles and their halos for the two-step (temporally blocked)
// update, and the tiles of the resident loop (build_loop_tiles).
//
// Chaining two updates of a cell without going back to memory (the paper's
// processor chaining, Sec. 7) needs, for a set of cells, the states of
// everything their two updates depend on.  Tile b is the contiguous range
// [b*T, min((b+1)*T, n)) of the current numbering (compact in space after a
// Hilbert renumbering).  Its first halo is every cell outside the tile that a
// tile cell has as a neighbour; its second halo every cell outside tile and
// first halo that a first-halo cell has as a neighbour.  The first step
// updates tile and first halo from states of tile and both halos; the second
// updates the tile from the first step's states of tile and first halo.
//
// Local numbering inside a tile: tile cells 0..nt-1 (nt cells in the tile),
// then the first halo (nt ..), then the second, each halo in ascending global
// id.  Neighbours are stored as 16-bit local ids; ghost faces keep their
// boundary code c < 0 as 0x10000 + c (0xFFFF wall, 0xFFFE far field, 0xFFFD
// extrapolation), so a tile with its halos holds at most 0xFFFD cells.
// Record of a tile cell: x = ids of faces 0 and 1, low half of y = id of
// face 2; bits 16 + 2k of y hold, for a face k whose neighbour is a cell of
// the same tile, the face of that neighbour that points back (the tile
// kernel that evaluates each face once writes the negated flux there).
#include <algorithm>
#include <cmath>
#include <exception>
#include <functional>
#include <thread>

#include "fv_internal.h"

namespace fv {

namespace {

constexpr int32_t kLocalLimit = 0xFFFD;  // first code used by ghost faces

uint32_t local_code(int32_t nb, int64_t t0, int64_t t1, int32_t nt, const std::vector<int32_t>& halo_pos,
                    const std::vector<int32_t>& stamp, int32_t b) {
  if (nb < 0) return (uint32_t)(0x10000 + nb);
  if (nb >= t0 && nb < t1) return (uint32_t)(nb - t0);
  if (stamp[nb] != b) throw Error{FV_EINVAL, "tile halo construction: neighbour outside the halo"};
  return (uint32_t)(nt + halo_pos[nb]);
}

}  // namespace

PairTiles build_pair_tiles(const HostMesh& m, int32_t tile) {
  if (tile < 1) throw Error{FV_EINVAL, "tile size must be positive"};
  if (m.n / tile >= INT32_MAX) throw Error{FV_EINVAL, "too many tiles"};
  PairTiles L;
  L.tile = tile;
  const int64_t n = m.n;
  L.n_tiles = (n + tile - 1) / tile;
  L.tile_info.assign(2 * (L.n_tiles + 1), 0);
  L.cell_ln.assign(2 * (size_t)n, 0u);
  // stamp[c] == b: c belongs to tile b's halos; halo_pos[c]: its position there
  std::vector<int32_t> stamp(n, -1);
  std::vector<int32_t> halo_pos(n, 0);
  std::vector<int32_t> h1, h2;
  for (int32_t b = 0; b < (int32_t)L.n_tiles; ++b) {
    const int64_t t0 = (int64_t)b * tile, t1 = std::min<int64_t>(t0 + tile, n);
    const int32_t nt = (int32_t)(t1 - t0);
    h1.clear();
    h2.clear();
    for (int64_t c = t0; c < t1; ++c)
      for (int k = 0; k < 3; ++k) {
        const int32_t x = m.nbr[3 * c + k];
        if (x >= 0 && (x < t0 || x >= t1) && stamp[x] != b) {
          stamp[x] = b;
          h1.push_back(x);
        }
      }
    std::sort(h1.begin(), h1.end());
    // cells of the first halo are marked; the second halo excludes them
    for (int32_t x : h1)
      for (int k = 0; k < 3; ++k) {
        const int32_t y = m.nbr[3 * (int64_t)x + k];
        if (y >= 0 && (y < t0 || y >= t1) && stamp[y] != b) {
          stamp[y] = b;
          h2.push_back(y);
        }
      }
    std::sort(h2.begin(), h2.end());
    const int64_t e_size = (int64_t)nt + (int64_t)h1.size() + (int64_t)h2.size();
    if (e_size > kLocalLimit)
      throw Error{FV_EINVAL, "a tile with its halos exceeds 65533 cells; renumber the cells "
                             "with a compact order (Hilbert) or use smaller tiles"};
    for (size_t j = 0; j < h1.size(); ++j) halo_pos[h1[j]] = (int32_t)j;
    for (size_t j = 0; j < h2.size(); ++j) halo_pos[h2[j]] = (int32_t)(h1.size() + j);
    const int64_t hs = (int64_t)L.halo_id.size();
    if (hs + (int64_t)h1.size() + (int64_t)h2.size() > INT32_MAX)
      throw Error{FV_EINVAL, "tile halos too large for 32-bit offsets"};
    L.tile_info[2 * b] = (int32_t)hs;
    L.tile_info[2 * b + 1] = (int32_t)h1.size();
    auto pack = [&](int64_t c, uint32_t* out, bool tile_cell) {
      const uint32_t a0 = local_code(m.nbr[3 * c], t0, t1, nt, halo_pos, stamp, b);
      const uint32_t a1 = local_code(m.nbr[3 * c + 1], t0, t1, nt, halo_pos, stamp, b);
      const uint32_t a2 = local_code(m.nbr[3 * c + 2], t0, t1, nt, halo_pos, stamp, b);
      out[0] = a0 | (a1 << 16);
      out[1] = a2;
      if (!tile_cell) return;
      for (int k = 0; k < 3; ++k) {
        const int32_t x = m.nbr[3 * c + k];
        if (x < t0 || x >= t1) continue;
        int kx = -1;
        for (int q = 0; q < 3; ++q)
          if (m.nbr[3 * (int64_t)x + q] == (int32_t)c && !(x == c && q == k) &&
              m.nrm[6 * (int64_t)x + 2 * q] == -m.nrm[6 * c + 2 * k] &&
              m.nrm[6 * (int64_t)x + 2 * q + 1] == -m.nrm[6 * c + 2 * k + 1])
            kx = q;
        if (kx < 0) throw Error{FV_EINVAL, "tile construction: the two sides of a face differ"};
        out[1] |= (uint32_t)kx << (16 + 2 * k);
      }
    };
    for (int64_t c = t0; c < t1; ++c) pack(c, &L.cell_ln[2 * c], true);
    // faces the tile evaluates once: every face of a tile cell, except those
    // whose other side is a tile cell of lower local id (or, for a cell
    // bordering itself, its own lower face)
    L.face_off.push_back((int32_t)(L.face_rec.size() / 2));
    for (int64_t c = t0; c < t1; ++c) {
      const uint32_t e = (uint32_t)(c - t0);
      const uint32_t w0 = L.cell_ln[2 * c], w1 = L.cell_ln[2 * c + 1];
      const uint32_t v[3] = {w0 & 0xFFFFu, w0 >> 16, w1 & 0xFFFFu};
      for (uint32_t q = 0; q < 3; ++q) {
        const uint32_t kq = (w1 >> (16 + 2 * q)) & 3u;
        if (v[q] < (uint32_t)nt && (v[q] < e || (v[q] == e && kq < q))) continue;
        L.face_rec.push_back(e | q << 16 | kq << 18);
        L.face_rec.push_back(v[q]);
      }
    }
    L.halo_ln.resize(2 * (hs + h1.size() + h2.size()), 0u);
    for (size_t j = 0; j < h1.size(); ++j) pack(h1[j], &L.halo_ln[2 * (hs + j)], false);
    L.halo_id.insert(L.halo_id.end(), h1.begin(), h1.end());
    L.halo_id.insert(L.halo_id.end(), h2.begin(), h2.end());
    L.e_cap = std::max<int32_t>(L.e_cap, (int32_t)e_size);
    L.t1_cap = std::max<int32_t>(L.t1_cap, nt + (int32_t)h1.size());
  }
  L.tile_info[2 * L.n_tiles] = (int32_t)L.halo_id.size();
  L.face_off.push_back((int32_t)(L.face_rec.size() / 2));
  if (L.face_rec.size() / 2 > (size_t)INT32_MAX) throw Error{FV_EINVAL, "too many tile faces"};
  return L;
}

namespace {

// Tiles [b0, b1) of build_step_tiles: their parts of tile_info (sizes only)
// and cell_ln in L, halo ids and faces in order in `part`.
struct TilePart {
  std::vector<int32_t> halo, faces_of;  // faces_of: faces of each tile
  std::vector<uint32_t> face_rec;
  int32_t t1_cap = 0, f_cap = 0;
};

// The cells of one tile's ring at a time and their places in it: an open table
// whose entries of earlier tiles are told by their stamp.
class RingTable {
 public:
  explicit RingTable(int32_t tile) {
    int bits = 4;
    while (((int64_t)1 << bits) < 8 * (int64_t)tile) ++bits;  // three neighbours a cell at most
    shift_ = 32 - bits;
    slots_.resize((size_t)1 << bits);
  }
  void next_tile() { ++now_; }
  // The place of cell x; `fresh` where it was not there (its place is then unset).
  int32_t& at(int32_t x, bool& fresh) {
    const uint32_t mask = (uint32_t)slots_.size() - 1u;
    uint32_t k = ((uint32_t)x * 2654435761u) >> shift_;
    while (slots_[k].stamp == now_ && slots_[k].cell != x) k = (k + 1u) & mask;
    fresh = slots_[k].stamp != now_;
    if (fresh) slots_[k] = Slot{x, 0, now_};
    return slots_[k].place;
  }

 private:
  struct Slot {
    int32_t cell = 0, place = 0;
    int64_t stamp = -1;
  };
  std::vector<Slot> slots_;
  int shift_;
  int64_t now_ = 0;
};

void step_tile_range(const HostMesh& m, int32_t tile, bool faces, int32_t b0, int32_t b1,
                     PairTiles& L, TilePart& part) {
  std::vector<int32_t> ring;
  std::vector<uint32_t> ghosts;
  RingTable places((int32_t)std::min<int64_t>(tile, m.n));
  bool fresh = false;
  for (int32_t b = b0; b < b1; ++b) {
    const int64_t t0 = (int64_t)b * tile, t1 = std::min<int64_t>(t0 + tile, m.n);
    const int32_t nt = (int32_t)(t1 - t0);
    ring.clear();
    places.next_tile();
    for (int64_t j = 3 * t0; j < 3 * t1; ++j) {
      const int32_t x = m.nbr[j];
      if (x < 0 || (x >= t0 && x < t1)) continue;
      places.at(x, fresh);
      if (fresh) ring.push_back(x);
    }
    std::sort(ring.begin(), ring.end());
    for (size_t e = 0; e < ring.size(); ++e) places.at(ring[e], fresh) = nt + (int32_t)e;
    if (nt + (int64_t)ring.size() > kLocalLimit)
      throw Error{FV_EINVAL, "a tile with its halo exceeds 65533 cells; renumber the cells "
                             "with a compact order (Hilbert) or use smaller tiles"};
    L.tile_info[2 * b + 1] = (int32_t)ring.size();
    part.t1_cap = std::max(part.t1_cap, nt + (int32_t)ring.size());
    part.halo.insert(part.halo.end(), ring.begin(), ring.end());
    const size_t first_face = part.face_rec.size();
    for (int64_t c = t0; c < t1; ++c) {
      const uint32_t e = (uint32_t)(c - t0);
      uint32_t v[3], back[3] = {0u, 0u, 0u};
      for (int k = 0; k < 3; ++k) {
        const int32_t x = m.nbr[3 * c + k];
        if (x < 0) {
          v[k] = (uint32_t)(0x10000 + x);
        } else if (x < t0 || x >= t1) {
          v[k] = (uint32_t)places.at(x, fresh);
        } else {
          v[k] = (uint32_t)(x - t0);
          if (!faces) continue;
          int kx = -1;  // the face of x that points back
          for (int q = 0; q < 3; ++q)
            if (m.nbr[3 * (int64_t)x + q] == (int32_t)c && !(x == c && q == k) &&
                m.nrm[6 * (int64_t)x + 2 * q] == -m.nrm[6 * c + 2 * k] &&
                m.nrm[6 * (int64_t)x + 2 * q + 1] == -m.nrm[6 * c + 2 * k + 1])
              kx = q;
          if (kx < 0) throw Error{FV_EINVAL, "tile construction: the two sides of a face differ"};
          back[k] = (uint32_t)kx;
        }
      }
      L.cell_ln[2 * c] = v[0] | (v[1] << 16);
      L.cell_ln[2 * c + 1] = v[2] | back[0] << 16 | back[1] << 18 | back[2] << 20;
      if (!faces) continue;
      for (uint32_t q = 0; q < 3; ++q) {
        if (v[q] < (uint32_t)nt && (v[q] < e || (v[q] == e && back[q] < q))) continue;
        std::vector<uint32_t>& list = v[q] < (uint32_t)kLocalLimit ? part.face_rec : ghosts;
        list.push_back(e | q << 16 | back[q] << 18);
        list.push_back(v[q]);
      }
    }
    // boundary faces last, so that they fill warps of their own
    part.face_rec.insert(part.face_rec.end(), ghosts.begin(), ghosts.end());
    ghosts.clear();
    const int32_t nf = (int32_t)((part.face_rec.size() - first_face) / 2);
    part.faces_of.push_back(nf);
    part.f_cap = std::max(part.f_cap, nf);
    for (int32_t i = 0; i < nf; ++i) {
      const uint32_t w = part.face_rec[first_face + 2 * i], v = part.face_rec[first_face + 2 * i + 1];
      auto refer = [&](uint32_t cell, uint32_t face, uint32_t ref) {
        L.cell_ref[2 * (t0 + cell) + (face >> 1)] |= ref << (face == 1 ? 16 : 0);
      };
      refer(w & 0xFFFFu, (w >> 16) & 3u, (uint32_t)i);
      if (v < (uint32_t)nt) refer(v, (w >> 18) & 3u, (uint32_t)i | 0x8000u);
    }
  }
}

}  // namespace

int host_workers(int64_t cells) {
  return (int)std::max<int64_t>(
      1, std::min<int64_t>({cells / 3000, 16, (int64_t)std::thread::hardware_concurrency()}));
}

void on_host_threads(int workers, const std::function<void(int)>& work) {
  std::vector<std::exception_ptr> errors(workers);
  auto guarded = [&](int w) {
    try {
      work(w);
    } catch (...) {
      errors[w] = std::current_exception();
    }
  };
  std::vector<std::thread> threads;
  int started = 1;  // this thread takes the first part, and those no thread could be had for
  try {
    threads.reserve(workers);
    for (; started < workers; ++started) threads.emplace_back(guarded, started);
  } catch (const std::exception&) {
  }
  guarded(0);
  for (int w = started; w < workers; ++w) guarded(w);
  for (std::thread& t : threads) t.join();
  for (const std::exception_ptr& e : errors)
    if (e) std::rethrow_exception(e);
}

PairTiles build_step_tiles(const HostMesh& m, int32_t tile, bool faces) {
  if (tile < 1) throw Error{FV_EINVAL, "tile size must be positive"};
  if (faces && tile > 10000) throw Error{FV_EINVAL, "tile too large for 15-bit face references"};
  if (m.n / tile >= INT32_MAX) throw Error{FV_EINVAL, "too many tiles"};
  PairTiles L;
  L.tile = tile;
  L.n_tiles = (m.n + tile - 1) / tile;
  L.tile_info.assign(2 * (L.n_tiles + 1), 0);
  L.cell_ln.resize(2 * (size_t)m.n);
  if (faces) L.cell_ref.assign(2 * (size_t)m.n, 0u);
  // starting a thread takes some 50 us, a cell some 10 ns: the time falls until
  // the square root of their ratio (host_workers' many threads spent 0.8 ms on
  // being started for 60,000 cells)
  const int workers = std::min(host_workers(m.n), 1 + (int)std::sqrt((double)m.n / 5000.0));
  std::vector<TilePart> parts(workers);
  on_host_threads(workers, [&](int w) {
    step_tile_range(m, tile, faces, (int32_t)(L.n_tiles * w / workers),
                    (int32_t)(L.n_tiles * (w + 1) / workers), L, parts[w]);
  });
  size_t halos = 0, words = 0;
  for (const TilePart& p : parts) {
    halos += p.halo.size();
    words += p.face_rec.size();
  }
  if (halos > (size_t)INT32_MAX || words / 2 > (size_t)INT32_MAX)
    throw Error{FV_EINVAL, "tile halos too large for 32-bit offsets"};
  L.halo_id.reserve(halos);
  L.face_rec.reserve(words);
  int32_t hs = 0, fs = 0, b = 0;
  for (const TilePart& p : parts) {
    L.halo_id.insert(L.halo_id.end(), p.halo.begin(), p.halo.end());
    L.face_rec.insert(L.face_rec.end(), p.face_rec.begin(), p.face_rec.end());
    L.t1_cap = std::max(L.t1_cap, p.t1_cap);
    L.f_cap = std::max(L.f_cap, p.f_cap);
    for (int32_t f : p.faces_of) {
      L.tile_info[2 * b] = hs;
      hs += L.tile_info[2 * b + 1];
      ++b;
      if (faces) L.face_off.push_back(fs);
      fs += f;
    }
  }
  L.tile_info[2 * L.n_tiles] = hs;
  if (faces) L.face_off.push_back(fs);
  L.e_cap = L.t1_cap;
  return L;
}

LoopTiles build_loop_tiles(const HostMesh& m, int32_t tile) {
  const int64_t n = m.n;
  if (tile < 1 || n > INT32_MAX || (n + tile - 1) / tile >= 0xFFFF)
    throw Error{FV_EINVAL, "resident loop: bad tile size"};
  LoopTiles L;
  L.tile = L.cap = tile;
  L.n_tiles = (int32_t)((n + tile - 1) / tile);
  L.info.assign(4 * (size_t)L.n_tiles, 0);
  L.ord.resize((size_t)n);
  L.cell_ln.resize(2 * (size_t)n);
  std::vector<int32_t> pos((size_t)n);  // local position of every cell in its tile
  std::vector<int32_t> inner, ring;
  int32_t edge_cells = 0;
  for (int32_t b = 0; b < L.n_tiles; ++b) {
    const int32_t t0 = b * tile, t1 = (int32_t)std::min<int64_t>((int64_t)t0 + tile, n);
    auto outside = [&](int32_t x) { return x >= 0 && (x < t0 || x >= t1); };
    inner.clear();
    ring.clear();
    int32_t at = t0;
    for (int32_t c = t0; c < t1; ++c) {
      const int32_t* x = &m.nbr[3 * (size_t)c];
      if (!outside(x[0]) && !outside(x[1]) && !outside(x[2])) {
        inner.push_back(c);
        continue;
      }
      pos[c] = at - t0;
      L.ord[at++] = c;
      for (int k = 0; k < 3; ++k)
        if (outside(x[k])) ring.push_back(x[k]);
    }
    const int32_t edges = at - t0;
    for (int32_t c : inner) {
      pos[c] = at - t0;
      L.ord[at++] = c;
    }
    std::sort(ring.begin(), ring.end());
    ring.erase(std::unique(ring.begin(), ring.end()), ring.end());
    if (tile + (int64_t)ring.size() > kLocalLimit)
      throw Error{FV_EINVAL, "resident loop: a tile with its ring exceeds 65533 cells"};
    L.cap = std::max(L.cap, tile + (int32_t)ring.size());
    L.info[4 * b] = (int32_t)L.ring_id.size();
    L.info[4 * b + 1] = (int32_t)ring.size();
    L.info[4 * b + 2] = edges;
    L.info[4 * b + 3] = edge_cells;
    edge_cells += edges;
    L.ring_id.insert(L.ring_id.end(), ring.begin(), ring.end());
  }
  // the entry of cell c in tile b's ring
  auto entry = [&](int32_t b, int32_t c) {
    const auto r0 = L.ring_id.begin() + L.info[4 * b], r1 = r0 + L.info[4 * b + 1];
    return (uint32_t)(std::lower_bound(r0, r1, c) - r0);
  };
  L.push.assign(3 * (size_t)edge_cells, 0xFFFFFFFFu);
  for (int32_t p = 0; p < (int32_t)n; ++p) {
    const int32_t b = p / tile, t0 = b * tile, e = p - t0, c = L.ord[p];
    const int32_t* x = &m.nbr[3 * (size_t)c];
    uint32_t v[3];
    for (int k = 0; k < 3; ++k) {
      const int32_t bx = x[k] < 0 ? b : x[k] / tile;
      if (x[k] < 0) {
        v[k] = (uint32_t)(0x10000 + x[k]);
      } else if (bx == b) {
        v[k] = (uint32_t)pos[x[k]];
      } else {
        v[k] = (uint32_t)tile + entry(b, x[k]);
        bool sent = false;
        for (int q = 0; q < k; ++q) sent = sent || (x[q] >= 0 && x[q] / tile == bx);
        if (!sent)
          L.push[3 * (size_t)(L.info[4 * b + 3] + e) + k] = (uint32_t)bx << 16 | entry(bx, c);
      }
    }
    L.cell_ln[2 * (size_t)p] = v[0] | (v[1] << 16);
    L.cell_ln[2 * (size_t)p + 1] = v[2];
  }
  return L;
}

}  // namespace fv
