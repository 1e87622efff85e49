// Neighbour rows: the Verlet list of a large replica on the mixed path (S.use_rows) as one row of partners per
// atom, and the static rows of its elastic network's soft springs.  One lane visits a row: it keeps the row's atom --
// position, parameters, force sum -- in registers and meets the partners one after the other, four at a time, so
// that a pair costs the loads and the fixed-point additions of one atom instead of two.  The forces are those of
// the pair list to the last bit: every contribution is split into the same two words, and the words are integers.
//
// What bounds it (2,030-atom ligand, per step of a block; by leaving parts out of a copy): of the list pass's 85k
// cycles about 44k go to evaluating and splitting the pairs (some 120 instructions each, four warps a scheduler), 10k
// to the additions, 7k to loading the partners and the rest to walking the rows; the pair list took 111k.  The
// springs stayed at 44k.  A rebuild takes 290k cycles against 640k.  Exit test, 1,024 replicas x 500 steps: 327 ->
// 245 ms.  Tried on top and left out: rows in shells of their distance at the build, visited as far as the
// largest displacement requires (22 % fewer partners, but the rebuild grew by half: 268 ms), forces kept in the
// accumulators to save their array (256 ms), lists rebuilt in a function of its own (290 ms).  Smaller, periodic and
// solvated systems keep the pair list: 220 atoms in a periodic box took 26.9 ms against 24.6 (seven tiles are too few
// rows for sixteen warps), the solvated ligand 380 against 325 (its passes spill).  So do replica sets whose rows would
// be longer than kRowPartners, and a replica that outgrows its rows on the way takes the pair list for the rest of the
// launch (segment.cu).  As rows of one pair each they took three times the pair list's time: globules at 100 atoms per
// nm^3 within 1.2 nm, 152 replicas x 20 steps, 1,024 atoms 5.5 -> 16.7 ms, 2,030 atoms 13.7 -> 39.4; at 40 per
// nm^3, whose rows fit, rows take 2.7 against 3.1 and 6.4 against 7.0 ms.
#pragma once
#include "state.cuh"

namespace grp {

// ---- the force sum of a row's atom in registers, added to the shared accumulators when the row ends
struct RowForce {
  int hi[3] = {0, 0, 0};
  unsigned int lo[3] = {0u, 0u, 0u};
  // minus a force, waiting for the partner's accumulators
  struct Other {
    Split s[3];
    __device__ __forceinline__ void add_to(const AccMixed &a, int j) const {
#pragma unroll
      for (int x = 0; x < 3; ++x) split_add(a.hi, a.lo, 3 * j + x, s[x]);
    }
  };
  // four forces at once: small ones (all but the closest contacts) split without conversions
  __device__ __forceinline__ void add(const V3<float> (&g)[4], Other (&o)[4], int *err) {
    bool small = true;
#pragma unroll
    for (int u = 0; u < 4; ++u) small = small && fabsf(g[u].x) + fabsf(g[u].y) + fabsf(g[u].z) < kSplitSmall;
    if (small) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float v[3] = {g[u].x, g[u].y, g[u].z};
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const Split p = to_split_small(v[x]);
          hi[x] += p.hi;
          lo[x] += p.lo;
          o[u].s[x] = to_split_small(-v[x]);
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float v[3] = {g[u].x, g[u].y, g[u].z};
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const Split p = to_split(v[x], err);
          hi[x] += p.hi;
          lo[x] += p.lo;
          o[u].s[x] = to_split(-v[x], err);
        }
      }
    }
  }
  __device__ __forceinline__ void flush(const AccMixed &a, int i) const {
#pragma unroll
    for (int x = 0; x < 3; ++x) split_add(a.hi, a.lo, 3 * i + x, Split{hi[x], lo[x]});
  }
};

// ---- the Verlet list of one replica
// Its memory is a pool of `cap` 32-bit words.
// The rows are sorted by length and taken 32 at a time, so that the 32 rows of a warp are about equally long; such a
// group holds its partners in blocks of 4 x 32 16-bit places, [block][lane][4], so that a lane's next four partners are one 8-byte load and a
// warp's are contiguous.  Blocks are worked off in chunks of up to `chunk` blocks of one group, so that the
// warps of the block get equal shares.  Tables at the end of the pool: the rows in order and their lengths,
// the groups' first blocks, and the chunks (group | blocks << 16 | first block in the group << 20, first block).
// While rows are built, those of a tile grow together in pieces of eight places for each of its 32 atoms
// ([lane][8], 512 bytes), taken one by one from the rest of the pool, up to 32 pieces (kRowPartners) a tile.
struct RowPool {
  int groups;  // of 32 rows
  int places;                // places of the blocks
  int pieces;                // pieces of the rows being built
  int scratch, chunks, first, order, lens, piece_of;  // word offsets: the pieces, and the tables
};
// 40 % of the pool holds the blocks, the rest the pieces: the pool has room for twice the pairs of the first configuration (or every pair).
__device__ __forceinline__ RowPool row_pool(const SysDev &S, int cap) {
  RowPool R;
  R.groups = (S.n + 31) >> 5;
  R.piece_of = cap - 16 * S.n_tiles;
  R.lens = R.piece_of - S.n;
  R.order = (R.lens - 2 * S.n) & ~1;
  R.first = R.order - R.groups - 1;
  R.chunks = (R.first - 2 * (cap / 160 + 1)) & ~3;
  const int room = max(0, R.chunks);
  R.scratch = (int)(0.4f * (float)room) & ~63;
  R.places = 2 * R.scratch;
  R.pieces = (room - R.scratch) / 128;
  return R;
}
struct RowList {
  const uint32_t *pool;
  int n, order, chunks;  // atoms, word offsets of the tables
  int n_chunks;
};

// Builds the rows of one replica: every non-excluded pair closer than cutoff + skin, on one of its atoms' rows
// (RowsDev::masks).  A warp takes a tile, tests the boxes of 32 partner tiles at once, and for each near one tests
// the 16 atoms j that can be on the lane's row (even lanes the odd ones and the other way round: two
// addresses for the whole warp), collecting a mask, and then writes the mask's atoms to the row.  (The pair-list
// build rotated j over the lanes and wrote through warp ballots: 640k cycles a build on the 2,030-atom
// ligand.)  False when a row or the blocks have no room (the caller then builds the pair list).  Called by every
// thread of the block; `bins` is scratch of 128 words, `taken` one more.
__device__ __forceinline__ bool build_rows(const SysDev &S, const RowsDev &W, const State<PathMixed> &st, const float *boxes, uint32_t *pool, int cap, RowList &L,
                           int *bins, int *taken) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, n = S.n;
  const RowPool R = row_pool(S, cap);
  uint16_t *rows = reinterpret_cast<uint16_t *>(pool + R.scratch), *piece_of = reinterpret_cast<uint16_t *>(pool + R.piece_of);
  uint32_t *lens = pool + R.lens, *first = pool + R.first;
  uint2 *order = reinterpret_cast<uint2 *>(pool + R.order);  // atom, length
  const float lc2 = S.list_cut2;
  for (int b = threadIdx.x; b < 128; b += blockDim.x) bins[b] = 0;
  if (threadIdx.x == 0) *taken = 0;
  __syncthreads();
  int over = 0;
  for (int I = warp; I < S.n_tiles; I += nwarps) {
    const int i = I * 32 + lane;
    const bool in = i < n;
    float xi[3] = {0.f, 0.f, 0.f};
    if (in) st.get_f32(i, xi);
    int cnt = 0, have = 0, mine = 0;  // have: pieces of this tile; mine: number of piece `lane`
    const int odd = (lane & 1) ^ 1;
    for (int e0 = 0; e0 < S.n_tiles; e0 += 32) {
      const int J = e0 + lane;
      bool near = false;
      if (J < S.n_tiles) {
        const float *ba = boxes + 6 * I, *bb = boxes + 6 * J;
        float g2 = 0.f;
        for (int x = 0; x < 3; ++x) {
          const float g = fmaxf(0.f, fmaxf(ba[x] - bb[x + 3], bb[x] - ba[x + 3]));
          g2 += g * g;
        }
        near = g2 < lc2;
      }
      unsigned todo = __ballot_sync(0xffffffffu, near);
      auto mask_of = [&](unsigned b) {
        return W.masks[((size_t)I * S.n_tiles + (e0 + __ffs(b) - 1)) * 32 + lane];
      };
      uint32_t next_mask = todo ? mask_of(todo) : 0u;
      for (; todo; todo &= todo - 1) {
        const int Jt = e0 + __ffs(todo) - 1, j0 = Jt * 32;
        const uint32_t mask = next_mask;
        if (todo & (todo - 1)) next_mask = mask_of(todo & (todo - 1));  // ahead of this tile's tests
        uint32_t hit = 0;
        auto meet = [&](int m) {
          float xj[3];
          st.get_f32(min(j0 + m, n - 1), xj);
          const float dx = xi[0] - xj[0], dy = xi[1] - xj[1], dz = xi[2] - xj[2];
          if (dx * dx + dy * dy + dz * dz < lc2) hit |= 1u << m;
        };
        if (Jt == I) {
#pragma unroll 8
          for (int m = 0; m < 32; ++m) meet(m);
        } else {
          // i + j is odd for the atoms of a higher tile, even for those of a lower one
          const int o = Jt > I ? odd : odd ^ 1;
#pragma unroll 8
          for (int m = 0; m < 32; m += 2) meet(m + o);
        }
        hit &= mask;
        const int need = __reduce_max_sync(0xffffffffu, cnt + __popc(hit));
        while (8 * have < need && !over) {
          int id = 0;
          if (lane == 0) id = atomicAdd(taken, 1);
          id = __shfl_sync(0xffffffffu, id, 0);
          if (have >= kRowPartners / 8 || id >= R.pieces) { over = 1; break; }
          if (lane == have) mine = id;
          ++have;
        }
        if (over) break;
        for (int left = __reduce_max_sync(0xffffffffu, __popc(hit)); left > 0; --left) {
          const int id = __shfl_sync(0xffffffffu, mine, (cnt >> 3) & 31);
          if (hit) {
            rows[(size_t)id * 256 + lane * 8 + (cnt & 7)] = (uint16_t)(j0 + __ffs(hit) - 1);
            hit &= hit - 1;
            ++cnt;
          }
        }
      }
      if (over) break;
    }
    if (over) break;
    if (lane < have) piece_of[I * 32 + lane] = (uint16_t)mine;
    if (in) {
      atomicAdd(&bins[min(cnt, 127)], 1);
      lens[i] = (uint32_t)cnt;
    }
  }
  if (__syncthreads_or(over)) return false;
  // counting sort of the rows by length, longest first
  if (warp == 0) {
    int c[4], s = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) { c[b] = bins[127 - (4 * lane + b)]; s += c[b]; }
    int incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    int at = incl - s;
#pragma unroll
    for (int b = 0; b < 4; ++b) { bins[127 - (4 * lane + b)] = at; at += c[b]; }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const uint32_t cnt = lens[i];
    order[atomicAdd(&bins[min((int)cnt, 127)], 1)] = make_uint2((uint32_t)i, cnt);
  }
  __syncthreads();
  // the groups' blocks and the chunks (one warp: a few dozen groups)
  if (warp == 0) {
    int total = 0;
    for (int g0 = 0; g0 < R.groups; g0 += 32) {
      const int g = g0 + lane;
      int longest = 0;
      if (g < R.groups) {
        const int r1 = min(32, n - 32 * g);
        for (int r = 0; r < r1; ++r) longest = max(longest, (int)order[32 * g + r].y);
      }
      const int nb = (longest + 3) >> 2;
      int incl = nb;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
      }
      if (g < R.groups) first[g] = (uint32_t)(total + incl - nb);
      total += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) {
      first[R.groups] = (uint32_t)total;
      bins[0] = total;
    }
    // about eight chunks per warp
    const int chunk = max(1, min(8, total / (8 * nwarps)));
    int nc = 0;
    __syncwarp();
    uint2 *table = reinterpret_cast<uint2 *>(pool + R.chunks);
    if (total * 128 <= R.places)
      for (int g0 = 0; g0 < R.groups; g0 += 32) {
        const int g = g0 + lane;
        const int f = g < R.groups ? (int)first[g] : 0, nb = g < R.groups ? (int)first[g + 1] - f : 0;
        const int mine = (nb + chunk - 1) / chunk;
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int x = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += x;
        }
        for (int c = 0; c < mine; ++c) {
          const int b0 = c * chunk;
          table[nc + incl - mine + c] = make_uint2((uint32_t)g | ((uint32_t)min(chunk, nb - b0) << 16) | ((uint32_t)b0 << 20),
                                                   (uint32_t)(f + b0));
        }
        nc += __shfl_sync(0xffffffffu, incl, 31);
      }
    if (lane == 0) bins[1] = nc;
  }
  __syncthreads();
  const int total = bins[0];
  L.n_chunks = bins[1];
  __syncthreads();
  if (total * 128 > R.places) return false;
  // the rows into their blocks
  for (int g = warp; g < R.groups; g += nwarps) {
    const int pos = 32 * g + lane;
    const uint2 w = pos < n ? order[pos] : make_uint2(0u, 0u);
    const uint16_t *row = rows + (w.x & 31u) * 8;
    const int src = (int)(w.x >> 5) * 32, cnt = (int)w.y, nb = (int)(first[g + 1] - first[g]);
    ushort4 *out = reinterpret_cast<ushort4 *>(pool) + (size_t)first[g] * 32 + lane;
#pragma unroll 4
    for (int b = 0; b < nb; ++b) {
      ushort4 x = make_ushort4(0, 0, 0, 0);
      if (4 * b < cnt) x = *reinterpret_cast<const ushort4 *>(row + (size_t)piece_of[src + (b >> 1)] * 256 + 4 * (b & 1));
      out[(size_t)b * 32] = x;
    }
  }
  __syncthreads();
  return true;
}

// The rows of a replica, shared out over the warps of the block chunk by chunk.  The visitor's begin(i),
// batch(partners, count) -- four places at a time, the first `count` of them filled (count <= 0: none) -- and
// end(any) are called by whole warps.  The next chunk's row and first partners are loaded ahead.
template <class V>
__device__ __forceinline__ void visit_rows(const RowList &L, V &&v) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int units = L.n_chunks;
  const uint2 *table = reinterpret_cast<const uint2 *>(L.pool + L.chunks);
  const ushort4 *blocks = reinterpret_cast<const ushort4 *>(L.pool) + lane;
  // loaded ahead: the table entry two units, the row and its first partners one unit
  const uint2 *order = reinterpret_cast<const uint2 *>(L.pool + L.order);
  auto entry = [&](int u) { return u < units ? table[u] : make_uint2(0u, 0u); };
  struct Unit {
    int i, cnt, nb, block;
    ushort4 j;
  };
  auto load = [&](int u, uint2 e) {
    Unit x{0, 0, 0, 0, make_ushort4(0, 0, 0, 0)};
    if (u >= units) return x;
    const int pos = 32 * (int)(e.x & 0xFFFFu) + lane;
    const uint2 w = pos < L.n ? order[pos] : make_uint2(0u, 0u);
    x.block = (int)e.y;
    x.j = blocks[(size_t)x.block * 32];
    x.nb = (int)((e.x >> 16) & 15u);
    x.i = (int)w.x;
    x.cnt = (int)w.y - 4 * (int)(e.x >> 20);
    return x;
  };
  Unit next = load(warp, entry(warp));
  uint2 after = entry(warp + nwarps);
  for (int u = warp; u < units; u += nwarps) {
    const Unit x = next;
    next = load(u + nwarps, after);
    after = entry(u + 2 * nwarps);
    v.begin(x.i);
    ushort4 j = x.j;
    for (int b = 0; b < x.nb; ++b) {
      const ushort4 now = j;
      if (b + 1 < x.nb) j = blocks[(size_t)(x.block + b + 1) * 32];
      v.batch(now, x.cnt - 4 * b);
    }
    v.end(x.cnt > 0);
  }
}

// ---- nonbonded forces of the rows (Lennard-Jones and Coulomb within the cutoff).  The four partners of a batch are loaded, then evaluated, then added, without branches
// between them, so that their chains overlap (one partner after the other, each behind the additions of the one
// before, the pass took 97k cycles per step on the 2,030-atom ligand against 111k for the pair list).  kE: with the
// pair energies (sampling steps).
__device__ __forceinline__ void row_params(const Params<PathMixed> &par, const Pos<PathMixed>::At &pa, int a, float &sh,
                                           float &se, float &qc) {
  sh = pa.h.w;  // as nb_params; the charges side by side where they fit in shared memory (a charge is one word at a
  se = pa.l.w;  // random atom, 32 cache lines of the global table for a warp)
  qc = par.qc ? par.qc[a] : par.atom[a].z;
}
template <int kRF, bool kE>
struct ListRow {
  using P = PathMixed;
  using T = float;
  const Pos<P> &pos;
  const Params<P> &par;
  const AccMixed &acc;
  long long &e_fix;
  int *err;
  T cut2;
  int i = 0;
  typename Pos<P>::At pi;
  T ash, ase, aqc;
  RowForce sum;
  __device__ __forceinline__ ListRow(float cutoff2, const Pos<P> &pos_, const Params<P> &par_, const AccMixed &a,
                                     long long &e, int *er)
      : pos(pos_), par(par_), acc(a), e_fix(e), err(er), cut2(cutoff2) {}
  __device__ __forceinline__ void begin(int at) {
    i = at;
    pi = pos.at(at);
    row_params(par, pi, at, ash, ase, aqc);
    sum = RowForce();
  }
  __device__ __forceinline__ void batch(ushort4 j4, int m) {
    const int J[4] = {m > 0 ? (int)j4.x : i, m > 1 ? (int)j4.y : i, m > 2 ? (int)j4.z : i, m > 3 ? (int)j4.w : i};
    typename Pos<P>::At pj[4];
    bool on[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      on[u] = u < m;
      pj[u].h = pos.qh[J[u]];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        // screen on the high words alone (their distance is within ~1e-6 of the double-single one): the
        // partners beyond the cutoff skip the low-word loads
        const V3<float> hd = {pi.h.x - pj[u].h.x, pi.h.y - pj[u].h.y, pi.h.z - pj[u].h.z};
        on[u] = on[u] && dot(hd, hd) <= cut2 * 1.0001f;
        pj[u].l = make_float4(0.f, 0.f, 0.f, 0.f);
        if (on[u]) pj[u].l = pos.ql[J[u]];
    }
    V3<T> f[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const V3<T> d = Pos<P>::diff(pi, pj[u]);
      T r2 = dot(d, d);
      on[u] = on[u] && r2 < cut2;
      r2 = on[u] ? r2 : T(1);
      T bsh, bse, bqc;
      row_params(par, pj[u], J[u], bsh, bse, bqc);
      const T sig = ash + bsh, eps = ase * bse, qq = aqc * bqc;
      const T inv_r2 = grcp(r2);
      const T s2 = sig * sig * inv_r2;
      const T s6 = s2 * s2 * s2;
      T g = pair_g<kRF>(par, eps, s6, qq, r2, inv_r2);
      g = on[u] ? g : T(0);
      f[u] = {g * d.x, g * d.y, g * d.z};
      if constexpr (kE)
        if (on[u]) e_fix += acc.efix(pair_e<kRF>(par, eps, s6, qq, r2, inv_r2), err);
    }
    RowForce::Other other[4];
    sum.add(f, other, err);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (on[u]) other[u].add_to(acc, J[u]);
  }
  __device__ __forceinline__ void end(bool any) {
    if (any) sum.flush(acc, i);
  }
};

// ---- soft springs on static rows: partners t .. t + 3 of atom i at [t / 4][i], 0xFFFF past an atom's last, their
// strengths and lengths beside them; the host gives each spring to the atom with the shorter row, so the rows of
// all atoms are about equally long.  A warp takes a tile; the next block's places are loaded ahead, across tiles.
// Stiff bonds, whose length needs double-single arithmetic, stay in a list of their own.
__device__ __forceinline__ void spring_rows(const SysDev &S, const RowsDev &W, const Pos<PathMixed> &pos, const Params<PathMixed> &par,
                                            const AccMixed &acc, bool want_e, long long &e_fix, int *err) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, n = S.n;
  for (int I = warp; I < S.n_tiles; I += nwarps) {
    const int i = I * 32 + lane, nb = (W.spring_rows[I] + 3) >> 2, ic = i < n ? i : n - 1;
    if (nb == 0) continue;
    RowForce sum;
    const float4 qi = pos.qh[ic];  // the high words suffice, as in bond_eval
    ushort4 next = __ldg(W.spring_j + ic);
    float4 nka = __ldg(W.spring_f + 2 * (size_t)ic), nkb = __ldg(W.spring_f + 2 * (size_t)ic + 1);
    for (int b = 0; b < nb; ++b) {
      const ushort4 j4 = next;
      const float4 ka = nka, kb = nkb;
      const size_t at = (size_t)b * n + ic;
      if (b + 1 < nb) {
        next = __ldg(W.spring_j + at + n);
        nka = __ldg(W.spring_f + 2 * (at + n));
        nkb = __ldg(W.spring_f + 2 * (at + n) + 1);
      }
      const float k[4] = {ka.x, ka.z, kb.x, kb.z}, r0[4] = {ka.y, ka.w, kb.y, kb.w};
      const int J[4] = {j4.x, j4.y, j4.z, j4.w};
      V3<float> d[4], f[4];
      bool on[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        on[u] = J[u] != 0xFFFF && i < n;
        const float4 qj = pos.qh[on[u] ? J[u] : ic];
        d[u] = {qi.x - qj.x, qi.y - qj.y, qi.z - qj.z};
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float r2 = dot(d[u], d[u]);
        r2 = on[u] ? r2 : 1.f;
        const float r = gsqrt(r2), dr = r - r0[u];
        float g = -gdiv(k[u] * dr, r);
        g = on[u] ? g : 0.f;
        f[u] = {g * d[u].x, g * d[u].y, g * d[u].z};
        if (want_e && on[u]) e_fix += acc.efix(0.5f * k[u] * dr * dr, err);
      }
      RowForce::Other other[4];
      sum.add(f, other, err);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (on[u]) other[u].add_to(acc, J[u]);
    }
    if (i < n) sum.flush(acc, i);
  }
  for (int t = threadIdx.x; t < W.n_stiff; t += blockDim.x) {
    const int b = W.stiff[t];
    const int2 ij = S.bond_ij[b];
    bond_term<PathMixed>(pos, par, b, ij.x, ij.y, acc, want_e, e_fix, err);
  }
}

}  // namespace grp
