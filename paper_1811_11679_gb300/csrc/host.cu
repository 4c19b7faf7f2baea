// host.cu -- the C ABI (include/hande.h): context set-up, system tables, device
// memory, CUDA-graph capture of one iteration, deterministic-space selection,
// estimator records and walker-list transfer.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <functional>
#include <new>
#include <string>
#include <vector>

#include "engine.h"
#include "host_util.h"

using namespace hande;

namespace {

const double kPi = 3.14159265358979323846;

void release_all(Engine& E) {
  learner_release(E);
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b)
      for (cudaGraphExec_t* g : {&E.graph[a][b], &E.graph_n[a][b]})
        if (*g) {
          cudaGraphExecDestroy(*g);
          *g = nullptr;
        }
  cudaStreamSynchronize(E.stream);
  for (auto& blk : E.blocks) {
    if (E.has_alloc) E.alloc.free(blk.first, blk.second, E.alloc.user);
    else cudaFree(blk.first);
  }
  E.blocks.clear();
  if (E.cap_stream) {
    cudaStreamDestroy(E.cap_stream);
    E.cap_stream = nullptr;
  }
  if (E.aux_stream) {
    cudaStreamDestroy(E.aux_stream);
    E.aux_stream = nullptr;
  }
  E.host.release();
  if (E.ev_fork) cudaEventDestroy(E.ev_fork);
  if (E.ev_join) cudaEventDestroy(E.ev_join);
  E.ev_fork = E.ev_join = nullptr;
}

// ---------------------------------------------------------------- system tables
struct HostTables {
  std::vector<int4> kvec;
  std::vector<int16_t> klookup;
  std::vector<double> h1, eri_packed;
  std::vector<int4> hb_pair;     // {start, len, guide offset, guide bits}
  std::vector<uint16_t> hb_ab;   // a | b << 8
  std::vector<double> hb_v;      // <pq||ab> (signed)
  std::vector<uint64_t> hb_cum;
  std::vector<double> hb_inv;    // inv_b = 2^64 / width (1 for a one-entry table)
  std::vector<ulonglong2> hb_ent;
  std::vector<uint16_t> pair_ij;
  std::vector<double> single_g;
  std::vector<uint16_t> hb_guide;
  std::vector<double> orb_diag, pair_diag;
};

inline size_t tri_h(size_t p, size_t q) { return p >= q ? p * (p + 1) / 2 + q : q * (q + 1) / 2 + p; }

// Hubbard hops: z per site, nbr[site z + k] (-1 = none).  Chain (ndim 0): hop 0
// to s + 1, hop 1 to s - 1, wrapped if periodic.  Lattice (ndim d): sites are
// the integer points whose coordinates in the basis of the lattice vectors
// (Cramer's rule, exact in integers) lie in [0, 1)^d, ordered lexicographically
// (checkerboard-interleaved for a bipartite cell);
// hop k moves by +e_{k/2} (k even) or -e_{k/2} (k odd) and is brought back
// into the cell by whole lattice vectors.  False if the lattice is degenerate,
// its cell does not hold norb sites, or a site's hops are not 2d distinct sites.
bool hubbard_hops(const hande_system& s, int& z, std::vector<int16_t>& nbr) {
  const int L = s.norb;
  if (s.ndim == 0) {
    z = 2;
    nbr.assign((size_t)2 * L, -1);
    for (int i = 0; i < L; ++i) {
      int right = i + 1, left = i - 1;
      if (s.periodic) {
        right = right == L ? 0 : right;
        left = left < 0 ? L - 1 : left;
      }
      nbr[2 * i] = (int16_t)(right < L ? right : -1);
      nbr[2 * i + 1] = (int16_t)(left >= 0 ? left : -1);
    }
    return true;
  }
  const int d = s.ndim;
  if (d < 1 || d > 3) return false;
  // lattice matrix padded with the identity; coordinates c of a point r in the
  // lattice basis: c_k = det(A with row k replaced by r) / det(A)
  int64_t A[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
  for (int i = 0; i < d; ++i)
    for (int j = 0; j < d; ++j) A[i][j] = s.lattice[3 * i + j];
  auto det3 = [](const int64_t M[3][3]) {
    return M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1]) - M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0]) +
           M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
  };
  const int64_t det = det3(A);
  if (det == 0 || (det < 0 ? -det : det) != L) return false;
  auto numer = [&](const int64_t r[3], int k) {   // det with row k replaced by r
    int64_t M[3][3];
    std::memcpy(M, A, sizeof M);
    for (int j = 0; j < 3; ++j) M[k][j] = r[j];
    return det3(M);
  };
  auto in_cell = [&](const int64_t r[3]) {
    for (int k = 0; k < d; ++k) {
      int64_t num = numer(r, k);
      if (det < 0) num = -num;
      const int64_t D = det < 0 ? -det : det;
      if (num < 0 || num >= D) return false;
    }
    return true;
  };
  // bounding box of the cell's corners
  int64_t lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
  for (int m = 0; m < (1 << d); ++m)
    for (int j = 0; j < d; ++j) {
      int64_t v = 0;
      for (int i = 0; i < d; ++i)
        if ((m >> i) & 1) v += A[i][j];
      lo[j] = std::min(lo[j], v);
      hi[j] = std::max(hi[j], v);
    }
  std::vector<std::array<int64_t, 3>> site;
  for (int64_t x = lo[0]; x <= hi[0]; ++x)
    for (int64_t y = lo[1]; y <= hi[1]; ++y)
      for (int64_t w = lo[2]; w <= hi[2]; ++w) {
        const int64_t r[3] = {x, y, w};
        if (in_cell(r)) site.push_back({x, y, w});
      }
  if ((int64_t)site.size() != L) return false;
  // checkerboard order for a bipartite cell (every lattice vector has an even
  // coordinate sum, equal halves): even-parity and odd-parity sites alternate,
  // each half lexicographic, so even indices form one sublattice
  bool bipartite = L % 2 == 0;
  for (int i = 0; i < d; ++i) bipartite = bipartite && ((A[i][0] + A[i][1] + A[i][2]) & 1) == 0;
  if (bipartite) {
    std::vector<std::array<int64_t, 3>> half[2];
    for (const auto& r : site) half[(r[0] + r[1] + r[2]) & 1].push_back(r);
    if (half[0].size() == half[1].size()) {
      for (size_t i = 0; i < half[0].size(); ++i) {
        site[2 * i] = half[0][i];
        site[2 * i + 1] = half[1][i];
      }
    }
  }
  z = 2 * d;
  nbr.assign((size_t)z * L, -1);
  const int64_t D = det < 0 ? -det : det;
  for (int i = 0; i < L; ++i)
    for (int k = 0; k < z; ++k) {
      int64_t r[3] = {site[i][0], site[i][1], site[i][2]};
      r[k >> 1] += (k & 1) ? -1 : 1;
      // subtract floor(c) whole lattice vectors
      int64_t shift[3] = {0, 0, 0};
      for (int q = 0; q < d; ++q) {
        int64_t num = numer(r, q);
        if (det < 0) num = -num;
        shift[q] = num >= 0 ? num / D : -((-num + D - 1) / D);
      }
      for (int q = 0; q < d; ++q)
        for (int j = 0; j < d; ++j) r[j] -= shift[q] * A[q][j];
      int t = -1;
      for (int j = 0; j < L; ++j)
        if (site[j][0] == r[0] && site[j][1] == r[1] && site[j][2] == r[2]) t = j;
      if (t < 0 || t == i) return false;
      for (int k2 = 0; k2 < k; ++k2)
        if (nbr[(size_t)i * z + k2] == t) return false;
      nbr[(size_t)i * z + k] = (int16_t)t;
    }
  return true;
}

// plane waves n in Z^3 ordered by (|n|^2, nx, ny, nz); the first norb are the basis
void build_ueg(const hande_system& s, SysDev& sd, HostTables& T) {
  struct PW {
    int n2, x, y, z;
  };
  int R = 1;
  std::vector<PW> pts;
  for (;;) {
    pts.clear();
    for (int x = -R; x <= R; ++x)
      for (int y = -R; y <= R; ++y)
        for (int z = -R; z <= R; ++z) {
          int n2 = x * x + y * y + z * z;
          if (n2 <= R * R) pts.push_back({n2, x, y, z});
        }
    if ((int)pts.size() > s.norb) break;
    ++R;
  }
  std::sort(pts.begin(), pts.end(), [](const PW& a, const PW& b) {
    if (a.n2 != b.n2) return a.n2 < b.n2;
    if (a.x != b.x) return a.x < b.x;
    if (a.y != b.y) return a.y < b.y;
    return a.z < b.z;
  });
  int nmax = 0;
  T.kvec.resize(s.norb);
  for (int i = 0; i < s.norb; ++i) {
    T.kvec[i] = make_int4(pts[i].x, pts[i].y, pts[i].z, pts[i].n2);
    nmax = std::max(nmax, std::max(std::abs(pts[i].x), std::max(std::abs(pts[i].y), std::abs(pts[i].z))));
  }
  int side = 2 * nmax + 1;
  T.klookup.assign((size_t)side * side * side, (int16_t)-1);
  for (int i = 0; i < s.norb; ++i)
    T.klookup[((size_t)(T.kvec[i].x + nmax) * side + (T.kvec[i].y + nmax)) * side + (T.kvec[i].z + nmax)] = (int16_t)i;
  sd.nmax = nmax;
  sd.side = side;
  // Omega = (4 pi / 3) rs^3 N, L = Omega^(1/3); 4 pi / (Omega (2 pi / L)^2 m) = 1 / (pi L m)
  const int nel = s.nalpha + s.nbeta;
  double box = s.rs * cbrt(4.0 * kPi * (double)nel / 3.0);
  sd.vfac = 1.0 / (kPi * box);
  double kf = 2.0 * kPi / box;
  sd.kfac = 0.5 * (kf * kf);
  // diagonal tables: kinetic |k|^2/2 per orbital, exchange kernel per orbital pair
  T.orb_diag.resize(s.norb);
  T.pair_diag.assign((size_t)s.norb * s.norb, 0.0);
  for (int i = 0; i < s.norb; ++i) {
    T.orb_diag[i] = sd.kfac * (double)T.kvec[i].w;
    for (int j = 0; j < s.norb; ++j) {
      int dx = T.kvec[i].x - T.kvec[j].x, dy = T.kvec[i].y - T.kvec[j].y, dz = T.kvec[i].z - T.kvec[j].z;
      int m = dx * dx + dy * dy + dz * dz;
      if (m > 0) T.pair_diag[(size_t)i * s.norb + j] = sd.vfac / (double)m;
    }
  }
}

// floor(x y 2^32) (half = false) or floor(x y 2^32 + 1/2) (half = true) of the
// exact product of two non-negative finite doubles, saturated at 2^62 (the
// device computes the same in fixed_amount)
uint64_t host_fixed_amount(double x, double y, bool half) {
  if (x == 0.0 || y == 0.0) return 0;
  uint64_t xb, yb;
  std::memcpy(&xb, &x, 8);
  std::memcpy(&yb, &y, 8);
  int ex = (int)(xb >> 52), ey = (int)(yb >> 52);
  uint64_t mx = xb & ((1ull << 52) - 1), my = yb & ((1ull << 52) - 1);
  if (ex) mx |= 1ull << 52;
  else ex = 1;
  if (ey) my |= 1ull << 52;
  else ey = 1;
  const unsigned __int128 prod = (unsigned __int128)mx * my;   // x y 2^32 = prod 2^(ex + ey - 2118)
  const int e = ex + ey - 2118;
  const uint64_t cap = 1ull << 62;
  if (e >= 0) {
    if (e >= 62 || (prod >> (62 - e)) != 0) return cap;
    return (uint64_t)(prod << e);
  }
  const int sh = -e;
  if (sh >= 120) return 0;
  const unsigned __int128 r = half ? ((prod >> (sh - 1)) + 1) >> 1 : prod >> sh;
  return r >= cap ? cap : (uint64_t)r;
}

double g_so(const std::vector<double>& eri, int n, int p, int q, int r, int t) {
  if (((p ^ q) & 1) || ((r ^ t) & 1)) return 0.0;
  size_t N = (size_t)n;
  return eri[(((size_t)(p >> 1) * N + (q >> 1)) * N + (r >> 1)) * N + (t >> 1)];
}

void build_molecule(const hande_system& s, const hande_qmc& q, SysDev& sd, HostTables& T) {
  const int n = s.norb;
  const size_t N = (size_t)n;
  T.h1.assign(s.h1, s.h1 + N * N);
  std::vector<double> eri(s.eri, s.eri + N * N * N * N);
  for (int p = 0; p < n; ++p)
    for (int r = 0; r < n; ++r)
      if (T.h1[p * N + r] != T.h1[r * N + p]) throw Fail{HANDE_ERR_INVALID, "h1 is not symmetric"};
  size_t npair = N * (N + 1) / 2;
  T.eri_packed.assign(npair * (npair + 1) / 2, 0.0);
  auto at = [&](size_t a, size_t b, size_t c, size_t d) { return eri[((a * N + b) * N + c) * N + d]; };
  for (size_t a = 0; a < N; ++a)
    for (size_t b = 0; b < N; ++b)
      for (size_t c = 0; c < N; ++c)
        for (size_t d = 0; d < N; ++d) {
          double v = at(a, b, c, d);
          if (v != at(b, a, c, d) || v != at(a, b, d, c) || v != at(c, d, a, b))
            throw Fail{HANDE_ERR_INVALID, "eri is not 8-fold symmetric"};
          T.eri_packed[tri_h(tri_h(a, b), tri_h(c, d))] = v;
        }
  sd.ecore = s.ecore;
  // diagonal tables: h_kk per spin orbital, (kk|ll) - (kl|lk) per spin-orbital pair
  const int nsp = 2 * n;
  T.orb_diag.resize(nsp);
  T.pair_diag.assign((size_t)nsp * nsp, 0.0);
  for (int p = 0; p < nsp; ++p) {
    T.orb_diag[p] = T.h1[(size_t)(p >> 1) * N + (p >> 1)];
    for (int q = 0; q < nsp; ++q) {
      double jv = at(p >> 1, p >> 1, q >> 1, q >> 1);
      double kv = ((p ^ q) & 1) ? 0.0 : at(p >> 1, q >> 1, q >> 1, p >> 1);
      T.pair_diag[(size_t)p * nsp + q] = jv - kv;
    }
  }
  // heat-bath tables: for each occupied pair p<q (index q(q-1)/2 + p), every
  // spin-allowed target pair a<b outside {p, q} with |<pq||ab>| > 0, in ascending
  // (a, b) order, as cumulative thresholds floor(2^64 S_k / S_total) made strictly
  // increasing; the last entry takes the remainder.
  const int ns = 2 * n;
  std::vector<int> hb_start((size_t)ns * (ns - 1) / 2, 0), hb_len((size_t)ns * (ns - 1) / 2, 0);
  for (int qq = 1; qq < ns; ++qq) {
    for (int pp = 0; pp < qq; ++pp) {
      const int idx = qq * (qq - 1) / 2 + pp;
      const int start = (int)T.hb_ab.size();
      std::vector<double> wts;
      for (int a = 0; a < ns; ++a) {
        for (int b = a + 1; b < ns; ++b) {
          if (a == pp || a == qq || b == pp || b == qq) continue;
          const bool direct = ((a & 1) == (pp & 1)) && ((b & 1) == (qq & 1));
          const bool swapped = ((a & 1) == (qq & 1)) && ((b & 1) == (pp & 1));
          if (!direct && !swapped) continue;
          double v = g_so(eri, n, pp, a, qq, b) - g_so(eri, n, pp, b, qq, a);
          double w = std::fabs(v);
          if (!(w > 0.0)) continue;
          T.hb_ab.push_back((uint16_t)(a | (b << 8)));
          T.hb_v.push_back(v);
          T.hb_cum.push_back(0);
          T.hb_inv.push_back(1.0);
          wts.push_back(w);
        }
      }
      const int len = (int)wts.size();
      hb_start[idx] = start;
      hb_len[idx] = len;
      if (len > 0) {
        std::vector<double> run(len);
        double acc = 0.0;
        for (int k = 0; k < len; ++k) {
          acc = acc + wts[k];
          run[k] = acc;
        }
        uint64_t last = 0;
        for (int k = 0; k + 1 < len; ++k) {
          double frac = run[k] / acc;
          uint64_t c = frac >= 1.0 ? ~0ull : (uint64_t)(frac * 18446744073709551616.0);
          if (c <= last) c = last + 1;
          T.hb_cum[start + k] = c;
          last = c;
        }
        T.hb_cum[start + len - 1] = ~0ull;
        // reciprocal of each entry's probability width / 2^64
        if (len > 1) {
          uint64_t prev = 0;
          for (int k = 0; k < len; ++k) {
            uint64_t width = (k + 1 == len) ? (0ull - prev) : (T.hb_cum[start + k] - prev);
            T.hb_inv[start + k] = 18446744073709551616.0 / (double)width;
            prev = T.hb_cum[start + k];
          }
        }
      }
    }
  }
  // single-excitation terms (ia|kk) - (ik|ka) over spin orbitals (zero unless spin(i) = spin(a))
  T.single_g.assign((size_t)ns * ns * ns, 0.0);
  for (int i = 0; i < ns; ++i)
    for (int a = 0; a < ns; ++a) {
      if ((i ^ a) & 1) continue;
      for (int k = 0; k < ns; ++k)
        T.single_g[((size_t)i * ns + a) * ns + k] = g_so(eri, n, i, a, k, k) - g_so(eri, n, i, k, k, a);
    }
  // guide of every heat-bath table: 2^g buckets with 2^g >= 2 len; for
  // t = 0 .. 2^g the first entry (among the first len - 1) whose threshold
  // exceeds t 2^(64-g), else len - 1
  T.hb_pair.assign(hb_start.size(), make_int4(0, 0, 0, 1));
  for (size_t idx = 0; idx < hb_start.size(); ++idx) {
    const int start = hb_start[idx], len = hb_len[idx];
    if (len > 65535) throw Fail{HANDE_ERR_INVALID, "heat-bath table too long"};
    if (len == 0) continue;
    int g = 1;
    while ((1 << g) < 2 * len) ++g;
    const int goff = (int)T.hb_guide.size();
    T.hb_pair[idx] = make_int4(start, len, goff, g);
    int k = 0;
    for (uint64_t t = 0; t <= (1ull << g); ++t) {
      if (t < (1ull << g)) {
        const uint64_t bound = t << (64 - g);
        while (k < len - 1 && !(T.hb_cum[start + k] > bound)) ++k;
      } else {
        k = len - 1;
      }
      T.hb_guide.push_back((uint16_t)k);
    }
  }
  sd.psingle_thr = (uint32_t)llrint(q.p_single * 4294967296.0);
  sd.p_single = (double)sd.psingle_thr * 0x1p-32;
  sd.p_double = (double)(4294967296ull - sd.psingle_thr) * 0x1p-32;
}

template <typename T>
T* upload(Engine& E, const std::vector<T>& v) {
  if (v.empty()) return nullptr;
  T* d = dalloc<T>(E, v.size());
  CK(cudaMemcpyAsync(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, E.stream));
  return d;
}

// The time step and every factor of the spawn weight that contains it:
// (tau inv_a) for each generator and the heat-bath entries' fixed-point amounts
// of |<pq||ab>| ((tau inv_a) inv_b), uploaded when `to_device`.
void set_tau(Engine& E, double tau, bool to_device) {
  SysDev& sd = E.P.sys;
  E.P.tau = tau;
  sd.c_hub = tau * sd.inv_hub;
  sd.c_ueg[0] = tau * sd.inv_ueg[0];
  sd.c_ueg[1] = tau * sd.inv_ueg[1];
  sd.c_single[0] = tau * sd.inv_single[0];
  sd.c_single[1] = tau * sd.inv_single[1];
  sd.c_tab = tau * sd.inv_tab;
  const double c_double = tau * E.inv_double;
  for (size_t k = 0; k < E.hb_ent.size(); ++k)
    E.hb_ent[k].x = host_fixed_amount(std::fabs(E.hb_v[k]), c_double * E.hb_inv[k], sd.half != 0);
  if (to_device && !E.hb_ent.empty())
    CK(cudaMemcpyAsync(const_cast<ulonglong2*>(sd.hb_ent), E.hb_ent.data(), E.hb_ent.size() * sizeof(ulonglong2),
                       cudaMemcpyHostToDevice, E.stream));
}

// The device state in the host block, after the stream's work (and after any
// copies the caller enqueued before this): one synchronisation.  Reading its
// words one by one cost a synchronisation each, about 10 us of the host's time.
constexpr size_t kHostState = (sizeof(DevState) + 63) & ~size_t(63);
char* host_block(Engine& E) { return E.host.get(kHostState + kPinRecords * sizeof(Record)); }
const DevState& read_state(Engine& E) {
  char* b = host_block(E);
  CK(cudaMemcpyAsync(b, E.P.st, sizeof(DevState), cudaMemcpyDeviceToHost, E.stream));
  CK(cudaStreamSynchronize(E.stream));
  return *reinterpret_cast<const DevState*>(b);
}
Record* pin_records(Engine& E) { return reinterpret_cast<Record*>(host_block(E) + kHostState); }

unsigned read_error(Engine& E) { return read_state(E).error; }

hande_status map_error(Engine& E, unsigned e) {
  if (!e) return HANDE_OK;
  E.failed = true;
  E.err_bits = e;
  if (e & ERR_OVERFLOW) {
    E.err = "population overflow (|N| reached 2^62 in fixed point)";
    return HANDE_ERR_OVERFLOW;
  }
  if (e & ERR_TIMEOUT) {
    E.err = "bounded device wait timed out (annihilation look-back)";
    return HANDE_ERR_TIMEOUT;
  }
  if (e & ERR_SPAWN_CAPACITY) E.err = "spawn capacity exceeded (raise spawn_capacity)";
  else if (e & ERR_TILE_CAPACITY) E.err = "annihilation tile capacity exceeded (too many distinct new determinants in one key range)";
  else if (e & ERR_STATE_CAPACITY) E.err = "walker-list capacity exceeded (raise state_capacity)";
  else E.err = "bucket capacity exceeded";
  return HANDE_ERR_CAPACITY;
}

void drop_graphs(Engine& E, int core);

// After an iteration while the time-step search runs: if the population has
// exceeded the target the search ends (tau stays); otherwise
// tau <- min(tau, 1 / R) with R the largest |H| / p_gen of any attempt so far.
void tau_search_step(Engine& E) {
  DevState hs;
  CK(cudaMemcpyAsync(&hs, E.P.st, sizeof hs, cudaMemcpyDeviceToHost, E.stream));
  CK(cudaStreamSynchronize(E.stream));
  if (hs.error) return;   // reported by the next synchronising call
  if (hs.vary) {
    E.tau_searching = false;
    E.P.tau_search = 0;
    E.P.sys.want_r = 0;
    drop_graphs(E, 0);
    drop_graphs(E, 1);
    return;
  }
  double r = 0.0;
  std::memcpy(&r, &hs.rmax_bits, 8);
  if (r > 0.0) {
    const double cand = 1.0 / r;
    if (cand < E.P.tau) {
      set_tau(E, cand, true);
      drop_graphs(E, 0);
      drop_graphs(E, 1);
    }
  }
}

// the captured graph of `iters` (1 or kGraphIters) iterations starting in list
// buffer cur
void ensure_graph(Engine& E, int cur, int core, int iters) {
  cudaGraphExec_t& slot = iters == 1 ? E.graph[cur][core] : E.graph_n[cur][core];
  if (slot) return;
  cudaGraph_t g = nullptr;
  CK(cudaStreamBeginCapture(E.cap_stream, cudaStreamCaptureModeThreadLocal));
  for (int i = 0; i < iters; ++i) E.ops.iteration(E, cur ^ (i & 1), core != 0, E.cap_stream, nullptr);
  cudaError_t launch_err = cudaGetLastError();
  CK(cudaStreamEndCapture(E.cap_stream, &g));
  if (launch_err != cudaSuccess) {
    cudaGraphDestroy(g);
    throw CudaError{launch_err, "kernel launch during capture"};
  }
  cudaGraphExec_t ex = nullptr;
  cudaError_t ie = cudaGraphInstantiate(&ex, g, 0);
  cudaGraphDestroy(g);
  CK(ie);
  slot = ex;
}

void drop_graphs(Engine& E, int core) {
  E.epoch += 1;   // the parameter block may have changed: batch graphs are rebuilt too
  for (int c = 0; c < 2; ++c)
    for (cudaGraphExec_t* g : {&E.graph[c][core], &E.graph_n[c][core]})
      if (*g) {
        cudaGraphExecDestroy(*g);
        *g = nullptr;
      }
}

// run the int64 scan machinery on natt[0..ndet[cur]) -> att_begin, total -> scan_total
void scan_natt(Engine& E, int cur) {
  Params& P = E.P;
  int64_t* n = st_field_i64(P.st, offsetof(DevState, ndet) + 8 * cur);
  k_scan_reduce<int64_t><<<kScanBlocks, kScanThreads, 0, E.stream>>>(P.natt, n, P.part, P.st);
  k_scan_partials_i64<<<1, 1024, 0, E.stream>>>(P.part, kScanBlocks, st_field_i64(P.st, offsetof(DevState, scan_total)),
                                                 P.st);
  k_scan_apply<int64_t><<<kScanBlocks, kScanThreads, 0, E.stream>>>(P.natt, P.att_begin, n, P.part, P.st);
  CK(cudaGetLastError());
}

// the core bit of every list flag (the iteration's other bits dropped), for
// hande_get_walkers
__global__ void k_core_flags(const uint8_t* in, uint8_t* out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = in[i] & F_CORE;
}

// Bucket-sizing statistics for the first iteration on a list set from the
// host: both "previous iteration" counts (spawns, distinct new keys) become the
// list's attempt bound, sum of ceil(|N_i|) walkers, so the buckets are sized
// as if every attempt spawned onto a new determinant.
__global__ void k_attempt_bound(const int64_t* pop, int64_t n, DevState* st) {
  __shared__ unsigned long long part[32];
  unsigned long long s = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = pop[i];
    const uint64_t m = (uint64_t)(p < 0 ? -p : p);
    s += (m + 0xffffffffull) >> 32;
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0ull;
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0 && s) {
      atomicAdd((unsigned long long*)&st->nspawn_prev, s);
      atomicAdd((unsigned long long*)&st->nuniq_prev, s);
    }
  }
}

int64_t read_i64(Engine& E, size_t off) {
  int64_t v = 0;
  CK(cudaMemcpyAsync(&v, (char*)E.P.st + off, 8, cudaMemcpyDeviceToHost, E.stream));
  CK(cudaStreamSynchronize(E.stream));
  return v;
}

void reserve_core(Engine& E, int64_t ncore);
void build_core_tables(Engine& E);

// Deterministic space "high": the reference plus the (size - 1) other
// determinants of largest |N| (ties by ascending key), then H' in CSR.
void select_core(Engine& E) {
  Params& P = E.P;
  const int cur = E.cur;
  const int64_t n = read_i64(E, offsetof(DevState, ndet) + 8 * cur);
  const int64_t want = (int64_t)E.core_size - 1;
  unsigned long long* hist = dalloc<unsigned long long>(E, 256);
  uint64_t vstar = 0;
  int64_t need_eq = INT64_MAX;
  if (want < n - 1) {  // otherwise every determinant is taken
    uint64_t mask = 0, prefix = 0;
    int64_t remaining = want;
    for (int shift = 56; shift >= 0; shift -= 8) {
      CK(cudaMemsetAsync(hist, 0, 256 * sizeof(unsigned long long), E.stream));
      E.ops.sel_hist(E, cur, shift, mask, prefix, hist, E.stream);
      unsigned long long h[256];
      CK(cudaMemcpyAsync(h, hist, sizeof h, cudaMemcpyDeviceToHost, E.stream));
      CK(cudaStreamSynchronize(E.stream));
      int d = 255;
      for (; d >= 0; --d) {
        if ((int64_t)h[d] >= remaining) break;
        remaining -= (int64_t)h[d];
      }
      if (d < 0) d = 0;
      prefix |= (uint64_t)d << shift;
      mask |= (uint64_t)255 << shift;
    }
    vstar = prefix;
    need_eq = remaining;
    if (want <= 0) {
      vstar = ~0ull;
      need_eq = 0;
    }
    E.ops.sel_flags(E, cur, vstar, need_eq, 0, E.stream);
    scan_natt(E, cur);
  }
  E.ops.sel_flags(E, cur, vstar, need_eq, 1, E.stream);
  scan_natt(E, cur);
  const int64_t ncore = read_i64(E, offsetof(DevState, scan_total));
  reserve_core(E, ncore);
  E.ops.sel_gather(E, cur, E.core_key, ncore, E.stream);
  P.ncore = (int)ncore;
  P.core_key = E.core_key;
  build_core_tables(E);
}

// device arrays of a deterministic space of ncore determinants
void reserve_core(Engine& E, int64_t ncore) {
  Params& P = E.P;
  if (ncore > E.ncore_cap) {
    E.core_key = dalloc<uint64_t>(E, (size_t)ncore * E.W);
    E.ncore_cap = ncore;
    P.core_pos = dalloc<int64_t>(E, ncore);
    P.core_delta = dalloc<int64_t>(E, ncore);
    P.core_x = dalloc<int64_t>(E, ncore);
    E.core_rowptr = dalloc<int64_t>(E, ncore + 1);
  }
}

// membership hash table and CSR of H' for the core keys in P.core_key (sorted,
// P.ncore of them, flagged in the list); the space is active afterwards
void build_core_tables(Engine& E) {
  Params& P = E.P;
  const int64_t ncore = P.ncore;
  // membership hash table: a power of two >= 4 ncore slots
  int64_t tsize = 64;
  while (tsize < 4 * ncore) tsize <<= 1;
  if (tsize > E.core_table_cap) {
    E.core_table = dalloc<uint32_t>(E, tsize);
    E.core_table_cap = tsize;
  }
  CK(cudaMemsetAsync(E.core_table, 0, (size_t)tsize * 4, E.stream));
  P.core_hmask = (uint32_t)(tsize - 1);
  P.core_hash = E.core_table;
  if (ncore > 0) E.ops.core_hash(E, E.core_table, E.stream);
  CK(cudaGetLastError());
  // CSR of H' restricted to the core
  int32_t* rowcnt = dalloc<int32_t>(E, ncore);
  E.ops.csr_count(E, rowcnt, E.stream);
  k_scan_small<<<1, 1024, 0, E.stream>>>(rowcnt, E.core_rowptr, (int)ncore);
  CK(cudaGetLastError());
  int64_t nnz = 0;
  CK(cudaMemcpyAsync(&nnz, E.core_rowptr + ncore, 8, cudaMemcpyDeviceToHost, E.stream));
  CK(cudaStreamSynchronize(E.stream));
  if (nnz > E.nnz_cap) {
    E.core_col = dalloc<int32_t>(E, nnz);
    E.core_val = dalloc<double>(E, nnz);
    E.nnz_cap = nnz;
  }
  P.core_rowptr = E.core_rowptr;
  P.core_col = E.core_col;
  P.core_val = E.core_val;
  E.ops.csr_fill(E, E.stream);
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(E.stream));
  drop_graphs(E, 1);
  E.core_active = true;
}

}  // namespace

// ================================================================= batch hooks
namespace hande {

// whether the replica can advance inside a batched graph (no per-iteration host
// work: no learned proposal, no running time-step search, no latched failure)
bool engine_batchable(const Engine& E) { return !E.failed && !E.learn && !E.tau_searching; }

// bookkeeping after a batched iteration; true if the deterministic space is
// due now (the caller orders E.stream after the iteration and calls
// engine_select_core)
bool engine_after_iteration(Engine& E) {
  E.cur ^= 1;
  E.host_iter += 1;
  return E.core_size > 0 && !E.core_active && E.core_start > 0 && E.host_iter == E.core_start;
}

hande_status engine_select_core(Engine& E);

}  // namespace hande

// ================================================================= C ABI
namespace {
hande_status run_guarded(Engine* E, const std::function<hande_status()>& body) {
  try {
    return body();
  } catch (const Fail& f) {
    if (E) {
      E->err = f.msg;
      if (f.code != HANDE_ERR_INVALID && f.code != HANDE_ERR_CAPACITY) E->failed = true;
    }
    return f.code;
  } catch (const CudaError& c) {
    if (E) {
      E->err = std::string(c.what) + ": " + cudaGetErrorString(c.e);
      E->failed = true;
    }
    return HANDE_ERR_CUDA;
  } catch (const std::bad_alloc&) {
    if (E) E->err = "host allocation failed";
    return HANDE_ERR_NOMEM;
  }
}
}  // namespace

namespace hande {
hande_status engine_select_core(Engine& E) {
  return run_guarded(&E, [&]() -> hande_status {
    hande_status es = map_error(E, read_error(E));
    if (es != HANDE_OK) return es;
    select_core(E);
    return HANDE_OK;
  });
}
}  // namespace hande

extern "C" {

hande_status hande_init_system(const hande_system* sys, const hande_qmc* qmc, const hande_allocator* allocator,
                               void* cuda_stream, hande_ctx** out) {
  if (!sys || !qmc || !out) return HANDE_ERR_INVALID;
  *out = nullptr;
  hande_ctx* ctx = new (std::nothrow) hande_ctx();
  if (!ctx) return HANDE_ERR_NOMEM;
  Engine& E = ctx->E;
  hande_status st = run_guarded(&E, [&]() -> hande_status {
    const hande_system& s = *sys;
    const hande_qmc& q = *qmc;
    // ---- validation
    if (s.key_words != 1 && s.key_words != 2 && s.key_words != 8) throw Fail{HANDE_ERR_INVALID, "key_words must be 1, 2 or 8"};
    if (s.kind < 0 || s.kind > 2) throw Fail{HANDE_ERR_INVALID, "unknown system kind"};
    if (s.norb < 1 || 2 * s.norb > 64 * s.key_words) throw Fail{HANDE_ERR_INVALID, "2*norb must fit in the key"};
    if (s.nalpha < 0 || s.nbeta < 0 || s.nalpha > s.norb || s.nbeta > s.norb || s.nalpha + s.nbeta < 2)
      throw Fail{HANDE_ERR_INVALID, "bad electron numbers"};
    if (s.kind == HANDE_HUBBARD) {
      if (s.ndim == 0 && s.periodic && s.norb < 3)
        throw Fail{HANDE_ERR_INVALID, "periodic Hubbard chain needs at least 3 sites"};
      if (s.nalpha > (s.norb + 1) / 2 || s.nbeta > s.norb / 2)
        throw Fail{HANDE_ERR_INVALID, "Hubbard reference needs nalpha <= ceil(L/2), nbeta <= floor(L/2)"};
    }
    if (s.kind == HANDE_MOLECULE && (!s.h1 || !s.eri || 2 * s.norb > 255))
      throw Fail{HANDE_ERR_INVALID, "molecule needs h1, eri and at most 127 orbitals"};
    if (s.kind == HANDE_UEG && !(s.rs > 0.0)) throw Fail{HANDE_ERR_INVALID, "UEG needs rs > 0"};
    if (!(q.tau > 0.0) || !(q.init_pop > 0.0)) throw Fail{HANDE_ERR_INVALID, "tau and init_pop must be positive"};
    if (q.semi_stoch_size > 0 && !q.real_amplitudes)
      throw Fail{HANDE_ERR_INVALID, "semi-stochastic propagation needs real amplitudes"};
    if (q.semi_stoch_size < 0 || q.semi_stoch_start < 0) throw Fail{HANDE_ERR_INVALID, "bad semi_stoch parameters"};
    if (q.real_amplitudes && !(q.spawn_cutoff >= 0.0)) throw Fail{HANDE_ERR_INVALID, "bad spawn_cutoff"};
    if (s.kind == HANDE_MOLECULE && !(q.p_single >= 0.0 && q.p_single < 1.0))
      throw Fail{HANDE_ERR_INVALID, "p_single must be in [0, 1)"};
    if (q.excit_gen != 0 && !(q.excit_gen == 1 && s.kind == HANDE_UEG))
      throw Fail{HANDE_ERR_INVALID, "excit_gen must be 0, or 1 (proposal table) for the UEG"};

    E.KW = s.key_words;
    E.kind = s.kind;
    E.nalpha = s.nalpha;
    E.nbeta = s.nbeta;
    E.stream = (cudaStream_t)cuda_stream;
    if (allocator && allocator->alloc && allocator->free) {
      E.alloc = *allocator;
      E.has_alloc = true;
    }
    // default annihilation: the flat hash path (32-bit list positions and spawn
    // indices), one warp per bucket for a list that does not fit those
    E.P.hash_merge = q.annihilation == 0 && q.state_capacity < ((int64_t)1 << 31) - 4 ? 1 : 0;
    E.W = E.KW == 8 && E.P.hash_merge && 2 * s.norb <= 192 ? 3 : E.KW;
    E.ops = E.W == 1 ? ops_w1(s.kind) : (E.W == 2 ? ops_w2(s.kind) : (E.W == 3 ? ops_w3(s.kind) : ops_w8(s.kind)));
    CK(cudaStreamCreateWithFlags(&E.cap_stream, cudaStreamNonBlocking));
    CK(cudaStreamCreateWithFlags(&E.aux_stream, cudaStreamNonBlocking));
    CK(cudaEventCreateWithFlags(&E.ev_fork, cudaEventDisableTiming));
    CK(cudaEventCreateWithFlags(&E.ev_join, cudaEventDisableTiming));

    Params& P = E.P;
    P.W = E.W;
    P.tau = q.tau;
    P.cutoff = q.spawn_cutoff;
    P.cutoff_fixed = q.spawn_cutoff * 4294967296.0 >= 4611686018427387904.0
                         ? kAmountMax
                         : (uint64_t)llrint(q.spawn_cutoff * 4294967296.0);
    P.zeta = q.shift_damping;
    P.real_amp = q.real_amplitudes ? 1 : 0;
    P.initiator = q.initiator ? 1 : 0;
    P.period = q.shift_period > 0 ? q.shift_period : 1;
    P.target_fixed = q.target_population * 4294967296.0 >= 9223372036854775807.0
                         ? INT64_MAX
                         : llrint(q.target_population * 4294967296.0);
    P.init_thr = q.initiator_threshold * 4294967296.0 >= 9223372036854775807.0
                     ? INT64_MAX
                     : llrint(q.initiator_threshold * 4294967296.0);
    P.seed = q.seed;
    P.replica = q.replica;
    P.max_det = q.state_capacity > 0 ? q.state_capacity : (int64_t)1 << 20;
    P.cap = (P.max_det + 3) & ~int64_t(3);
    P.scap = q.spawn_capacity > 0 ? q.spawn_capacity : (int64_t)1 << 21;
    if (P.scap >= ((int64_t)1 << 31)) throw Fail{HANDE_ERR_INVALID, "spawn_capacity must be below 2^31"};
    P.rec_cap = q.record_capacity > 0 ? q.record_capacity : 1 << 16;
    // on-chip tile: distinct new keys (TC, a power of two for the bitonic sort) and
    // main-list entries (SM) per bucket
    if (q.annihilation < 0 || q.annihilation > 2) throw Fail{HANDE_ERR_INVALID, "annihilation must be 0, 1 or 2"};
    E.merge_warp = !P.hash_merge && q.annihilation != 1;
    // block tiles: sized so that four 256-thread CTAs share an SM for 64- and
    // 128-bit keys (two for 512-bit keys).  Warp path (three 8-warp CTAs per SM,
    // two for 512-bit keys): 128 staged new keys per warp and segments of
    // at most 192 entries (64 and 96 for 512-bit keys), buckets sized for 1.5 x
    // the staging in expected spawns (most land on listed entries) and for half
    // the staging in distinct new keys; the buckets it defers go to block tiles.
    P.tile_cap = E.KW == 8 ? 256 : 512;
    P.seg_max = E.merge_warp ? E.ops.merge_warp_main : (E.W == 1 ? 768 : (E.W == 2 ? 512 : 256));
    P.warp_cap = E.ops.merge_warp_new;
    if (q.tile_capacity > 0) {
      int tc = q.tile_capacity;
      if (tc < 64 || tc > P.tile_cap || (tc & (tc - 1)))
        throw Fail{HANDE_ERR_INVALID, "tile_capacity must be a power of two in [64, default]"};
      P.tile_cap = tc;
      P.seg_max = std::min(P.seg_max, tc);
      P.warp_cap = std::min(E.ops.merge_warp_new, tc);
    }
    P.bucket_spawns = E.merge_warp ? P.warp_cap * 3 / 2 : P.tile_cap / 2;
    P.bucket_new = E.merge_warp ? P.warp_cap / 2 : 0;
    E.core_size = q.semi_stoch_size;
    E.core_start = q.semi_stoch_start;

    // ---- reference determinant
    std::memset(P.d0, 0, sizeof P.d0);
    auto setbit = [&](int p) { P.d0[p >> 6] |= 1ull << (p & 63); };
    if (s.kind == HANDE_HUBBARD) {
      for (int k = 0; k < s.nalpha; ++k) setbit(2 * (2 * k));
      for (int k = 0; k < s.nbeta; ++k) setbit(2 * (2 * k + 1) + 1);
    } else {
      for (int k = 0; k < s.nalpha; ++k) setbit(2 * k);
      for (int k = 0; k < s.nbeta; ++k) setbit(2 * k + 1);
    }

    // ---- system tables
    SysDev& sd = P.sys;
    std::memset(&sd, 0, sizeof sd);
    sd.norb = s.norb;
    sd.nspin = 2 * s.norb;
    sd.nel = s.nalpha + s.nbeta;
    sd.L = s.norb;
    sd.periodic = s.periodic;
    sd.t = s.t;
    sd.U = s.U;
    HostTables T;
    std::vector<int16_t> hops;
    sd.z = 0;
    if (s.kind == HANDE_HUBBARD && !hubbard_hops(s, sd.z, hops))
      throw Fail{HANDE_ERR_INVALID, "Hubbard lattice: degenerate, |det| != norb, or hops not to distinct sites"};
    if (s.kind == HANDE_UEG) build_ueg(s, sd, T);
    if (s.kind == HANDE_MOLECULE) build_molecule(s, q, sd, T);
    {
      const int n = sd.nel;
      const double npairs = (double)((int64_t)n * (n - 1) / 2);
      // 1/p_gen = inv_a inv_b; the spawn-weight factors (tau inv_a) inv_b follow in set_tau
      sd.inv_hub = (double)sd.z * (double)n;
      sd.inv_ueg[0] = (npairs * (double)s.norb) / 2.0;
      sd.inv_ueg[1] = (npairs * (double)s.norb) / 1.0;
      sd.inv_single[0] = ((double)n * (double)(s.norb - s.nalpha)) / sd.p_single;
      sd.inv_single[1] = ((double)n * (double)(s.norb - s.nbeta)) / sd.p_single;
      sd.inv_tab = npairs;
      sd.half = q.real_amplitudes ? 1 : 0;
      E.inv_double = npairs / sd.p_double;
      // heat-bath entries: (a, b, sign) now, the amounts in set_tau
      E.hb_v = T.hb_v;
      E.hb_inv = T.hb_inv;
      E.hb_ent.resize(T.hb_ab.size());
      for (size_t k = 0; k < T.hb_ab.size(); ++k)
        E.hb_ent[k].y = (unsigned long long)T.hb_ab[k] | ((T.hb_v[k] < 0.0 ? 1ull : 0ull) << 16);
      set_tau(E, q.tau, false);
      T.hb_ent = E.hb_ent;
      // time-step search: |<pq||ab>| / p_gen = (|<pq||ab>| inv_a) inv_b per entry
      E.tau_search_on = E.tau_searching = q.tau_search != 0;
      E.P.tau_search = q.tau_search != 0 ? 1 : 0;
      sd.want_r = E.P.tau_search;
      if (q.tau_search && !T.hb_v.empty()) {
        std::vector<double> R(T.hb_v.size());
        for (size_t k = 0; k < R.size(); ++k) R[k] = (std::fabs(T.hb_v[k]) * E.inv_double) * T.hb_inv[k];
        sd.hb_R = upload(E, R);
      }
    }
    sd.kvec = upload(E, T.kvec);
    sd.klookup = upload(E, T.klookup);
    sd.h1 = upload(E, T.h1);
    sd.eri = upload(E, T.eri_packed);
    sd.hb_pair = upload(E, T.hb_pair);
    sd.hb_cum = upload(E, T.hb_cum);
    sd.hb_ent = upload(E, T.hb_ent);
    sd.hb_ab = upload(E, T.hb_ab);
    for (int j = 1; j < sd.nel; ++j)
      for (int i = 0; i < j; ++i) T.pair_ij.push_back((uint16_t)(i | (j << 8)));
    sd.pair_ij = upload(E, T.pair_ij);
    sd.single_g = upload(E, T.single_g);
    sd.hb_guide = upload(E, T.hb_guide);
    sd.orb_diag = upload(E, T.orb_diag);
    sd.pair_diag = upload(E, T.pair_diag);
    sd.nbr = upload(E, hops);
    sd.ptab_cum = nullptr;
    if (q.excit_gen == 1) proposal_init(E, T.kvec.data(), T.klookup.data(), sd.nmax, sd.side);

    // ---- device buffers
    const int64_t cap = P.cap, scap = P.scap;
    for (int b = 0; b < 2; ++b) {
      P.key[b] = dalloc<uint64_t>(E, (size_t)cap * E.KW);   // also stages keys of KW words
      P.pop[b] = dalloc<int64_t>(E, cap);
      P.hdiag[b] = dalloc<double>(E, cap);
      P.flags[b] = dalloc<uint8_t>(E, cap);
    }
    if (E.W > 2) P.fold = dalloc<uint64_t>(E, 2 * (size_t)cap);
    P.natt = dalloc<int64_t>(E, cap);
    P.att_begin = dalloc<int64_t>(E, cap);
    P.part = dalloc<int64_t>(E, kScanBlocks + 1);
    const size_t det_states = (size_t)(cap / kDetTile + 33);   // a short list has up to 32 smaller tiles
    P.det_state = dalloc<unsigned long long>(E, det_states);
    CK(cudaMemsetAsync(P.det_state, 0, det_states * sizeof(unsigned long long), E.stream));
    P.s_key = dalloc<uint64_t>(E, (size_t)scap * E.W);
    P.s_amt = dalloc<int64_t>(E, scap);
    P.s_meta = dalloc<uint64_t>(E, scap);
    P.b_key = dalloc<uint64_t>(E, (size_t)scap * E.W);
    P.b_amt = dalloc<int64_t>(E, scap);
    if (P.hash_merge) {
      const int64_t tiles = list_tiles(cap);
      P.hash_size = 1024;
      while (P.hash_size < 2 * (uint64_t)scap && P.hash_size < (1ull << 31)) P.hash_size <<= 1;
      P.hash_tab = dalloc<uint32_t>(E, P.hash_size);
      P.u_spawn = dalloc<uint32_t>(E, scap);
      P.u_rank = dalloc<uint32_t>(E, scap);
      P.n_pos = dalloc<uint32_t>(E, scap);
      P.n_order = dalloc<uint32_t>(E, scap);
      P.g_new = dalloc<uint32_t>(E, (tiles + 1) * kGroups);   // the det pass clears one tile ahead
      P.g_keep = dalloc<uint64_t>(E, tiles * kGroups);
      P.g_pre = dalloc<uint32_t>(E, tiles * kGroups);
      P.t_keep = dalloc<uint32_t>(E, tiles);
      P.t_base = dalloc<unsigned long long>(E, tiles);
      P.occ_draw = dalloc<uint32_t>(E, cap);
      P.core_move = dalloc<uint32_t>(E, cap);
      // (one allocation for the levels: twelve took 25 us of the 180 that creating and
      // destroying a small context takes)
      size_t ends = 0;
      for (int l = 1; l < kEndLevels && (cap >> (2 * l)) > 0; ++l) ends += (size_t)end_stride(cap, l) * E.W;
      uint64_t* end = dalloc<uint64_t>(E, ends);
      for (int l = 1; l < kEndLevels && (cap >> (2 * l)) > 0; ++l) {
        P.s_end[l] = end;
        end += (size_t)end_stride(cap, l) * E.W;
      }
      CK(cudaMemsetAsync(P.hash_tab, 0, P.hash_size * sizeof(uint32_t), E.stream));
    } else {
      P.b_flag = dalloc<uint8_t>(E, scap);
      P.bcount = dalloc<uint32_t>(E, cap);
      P.boff = dalloc<uint32_t>(E, cap);
      P.tile_state = dalloc<unsigned long long>(E, cap);
      P.split_key = dalloc<uint64_t>(E, (size_t)cap * E.W);
    }
    if (E.merge_warp) {
      P.tile_inc = dalloc<unsigned long long>(E, cap);
      P.mcap = cap + scap;   // >= main entries + spawns of one iteration
      P.m_key = dalloc<uint64_t>(E, (size_t)P.mcap * E.W);
      P.m_pop = dalloc<int64_t>(E, P.mcap);
      P.m_hd = dalloc<double>(E, P.mcap);
      P.m_flg = dalloc<uint8_t>(E, P.mcap);
    }
    P.st = dalloc<DevState>(E, 1);
    E.check_word = dalloc<unsigned>(E, 4);
    P.rec = dalloc<Record>(E, P.rec_cap);
    P.ncore = 0;

    // ---- launch geometry
    int dev = 0, nsm = 0;
    CK(cudaGetDevice(&dev));
    E.device = dev;
    CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    if (!P.hash_merge) {
      E.merge_smem_bytes = E.ops.merge_smem(P.tile_cap, P.seg_max);
      CK(cudaFuncSetAttribute(E.ops.merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)E.merge_smem_bytes));
      int per_sm = 0;
      CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, E.ops.merge_kernel, kMergeThreads,
                                                       E.merge_smem_bytes));
      if (per_sm < 1) throw Fail{HANDE_ERR_CUDA, "annihilation kernel does not fit on an SM"};
      E.merge_grid = per_sm * nsm;
    }
    if (E.merge_warp) {
      CK(cudaFuncSetAttribute(E.ops.merge_warp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)E.ops.merge_warp_smem));
      int wper = 0;
      CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&wper, E.ops.merge_warp_kernel, kMwThreads,
                                                       E.ops.merge_warp_smem));
      if (wper < 1) throw Fail{HANDE_ERR_CUDA, "warp annihilation kernel does not fit on an SM"};
      E.merge_warp_grid = wper * nsm;
    }
    CK(cudaFuncSetAttribute(E.ops.attempt_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                            (int)E.ops.attempt_smem));
    int att_per_sm = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&att_per_sm, E.ops.attempt_kernel, kAttemptThreads,
                                                     E.ops.attempt_smem));
    if (att_per_sm < 1) throw Fail{HANDE_ERR_CUDA, "spawning kernel does not fit on an SM"};
    E.attempt_grid = att_per_sm * nsm;

    // ---- initial state: init_pop walkers on the reference
    DevState hs;
    std::memset(&hs, 0, sizeof hs);
    hs.ndet[0] = 1;
    CK(cudaMemcpyAsync(P.st, &hs, sizeof hs, cudaMemcpyHostToDevice, E.stream));
    E.ops.eref(E, E.stream);
    for (int j = 0; j < E.W; ++j)
      CK(cudaMemcpyAsync(P.key[0] + (size_t)j * cap, &P.d0[j], 8, cudaMemcpyHostToDevice, E.stream));
    int64_t p0 = llrint(q.init_pop * 4294967296.0);
    double h0 = 0.0;
    uint8_t f0 = 0;
    CK(cudaMemcpyAsync(P.pop[0], &p0, 8, cudaMemcpyHostToDevice, E.stream));
    CK(cudaMemcpyAsync(P.hdiag[0], &h0, 8, cudaMemcpyHostToDevice, E.stream));
    CK(cudaMemcpyAsync(P.flags[0], &f0, 1, cudaMemcpyHostToDevice, E.stream));
    CK(cudaGetLastError());
    E.e_ref = 0.0;
    CK(cudaMemcpyAsync(&E.e_ref, (char*)P.st + offsetof(DevState, e_ref), 8, cudaMemcpyDeviceToHost, E.stream));
    CK(cudaStreamSynchronize(E.stream));
    E.cur = 0;
    if (E.core_size > 0 && E.core_start == 0) select_core(E);
    return HANDE_OK;
  });
  if (st != HANDE_OK) {
    release_all(E);
    delete ctx;
    return st;
  }
  *out = ctx;
  return HANDE_OK;
}

hande_status hande_iterate(hande_ctx* ctx, int n) {
  if (!ctx || n < 0) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    for (int k = 0; k < n; ++k) {
      int core = E.core_active ? 1 : 0;
      // several iterations per launch when no host work is due between them
      const bool core_due = E.core_size > 0 && !E.core_active && E.core_start > E.host_iter &&
                            E.core_start <= E.host_iter + kGraphIters;
      if (n - k >= kGraphIters && !(E.learn && learner_period(E) > 0) && !E.tau_searching && !core_due) {
        ensure_graph(E, E.cur, core, kGraphIters);
        CK(cudaGraphLaunch(E.graph_n[E.cur][core], E.stream));
        E.host_iter += kGraphIters;
        k += kGraphIters - 1;
        continue;
      }
      ensure_graph(E, E.cur, core, 1);
      CK(cudaGraphLaunch(E.graph[E.cur][core], E.stream));
      E.cur ^= 1;
      E.host_iter += 1;
      if (learner_due(E)) learner_step(E);
      if (E.tau_searching) tau_search_step(E);
      if (E.core_size > 0 && !E.core_active && E.core_start > 0 && E.host_iter == E.core_start) {
        hande_status es = map_error(E, read_error(E));
        if (es != HANDE_OK) return es;
        select_core(E);
      }
    }
    return HANDE_OK;
  });
}

hande_status hande_iterate_timed(hande_ctx* ctx, int n, float* phase_ms, int nphases) {
  if (!ctx || n < 0 || !phase_ms || nphases < kPhases) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    cudaEvent_t ev[kPhases + 1];
    for (int k = 0; k <= kPhases; ++k) CK(cudaEventCreate(&ev[k]));
    struct Cleanup {
      cudaEvent_t* e;
      ~Cleanup() {
        for (int k = 0; k <= kPhases; ++k) cudaEventDestroy(e[k]);
      }
    } cleanup{ev};
    for (int k = 0; k < kPhases; ++k) phase_ms[k] = 0.0f;
    for (int it = 0; it < n; ++it) {
      E.ops.iteration(E, E.cur, E.core_active, E.stream, ev);
      CK(cudaGetLastError());
      CK(cudaEventSynchronize(ev[kPhases]));
      for (int k = 0; k < kPhases; ++k) {
        float ms = 0.0f;
        CK(cudaEventElapsedTime(&ms, ev[k], ev[k + 1]));
        phase_ms[k] += ms;
      }
      E.cur ^= 1;
      E.host_iter += 1;
      if (E.core_size > 0 && !E.core_active && E.core_start > 0 && E.host_iter == E.core_start) {
        hande_status es = map_error(E, read_error(E));
        if (es != HANDE_OK) return es;
        select_core(E);
      }
    }
    return HANDE_OK;
  });
}

hande_status hande_synchronize(hande_ctx* ctx) {
  if (!ctx) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status { return map_error(E, read_error(E)); });
}

hande_status hande_estimators(hande_ctx* ctx, hande_estimate* out, int max, int* n_out) {
  if (!ctx || max < 0 || (max > 0 && !out)) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (n_out) *n_out = 0;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    bool lost = false;
    if (E.host_iter - E.fetched > E.P.rec_cap) {
      E.fetched = E.host_iter - E.P.rec_cap;
      lost = true;
    }
    const int64_t avail = E.host_iter - E.fetched;
    const int64_t m = std::min<int64_t>(avail, max);
    std::vector<Record> big;
    Record* tmp = pin_records(E);
    if (m > kPinRecords) {
      big.resize((size_t)m);
      tmp = big.data();
    }
    if (m > 0) {   // the ring's slots from the first unread one: at most two contiguous runs
      const int64_t first = E.fetched % E.P.rec_cap;
      const int64_t run = std::min<int64_t>(m, E.P.rec_cap - first);
      CK(cudaMemcpyAsync(tmp, E.P.rec + first, (size_t)run * sizeof(Record), cudaMemcpyDeviceToHost, E.stream));
      if (m > run)
        CK(cudaMemcpyAsync(tmp + run, E.P.rec, (size_t)(m - run) * sizeof(Record), cudaMemcpyDeviceToHost, E.stream));
    }
    hande_status es = map_error(E, read_error(E));   // synchronises; the records came before it
    if (es != HANDE_OK) return es;
    for (int64_t i = 0; i < m; ++i) {
      const Record& r = tmp[i];
      hande_estimate& o = out[i];
      o.iter = r.iter;
      o.shift = r.shift;
      o.nw_pre = r.nw_pre;
      o.n0 = r.n0;
      o.num_hi = r.num_hi;
      o.num_lo = r.num_lo;
      o.num = r.num;
      o.nw_post = r.nw_post;
      o.ndet = r.ndet;
      o.natt = r.natt;
      o.nspawn = r.nspawn;
      o.tau = r.tau;
    }
    E.fetched += m;
    if (n_out) *n_out = (int)m;
    if (lost) {
      E.err = "estimator records were overwritten before being fetched";
      return HANDE_ERR_CAPACITY;
    }
    return HANDE_OK;
  });
}

hande_status hande_get_walkers(hande_ctx* ctx, uint64_t* keys, int64_t* pops, double* hdiag, uint8_t* flags,
                               int64_t cap, int64_t* n) {
  if (!ctx || !n) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    const int cur = E.cur;
    const DevState& hs = read_state(E);
    const int64_t nd = hs.ndet[cur];
    hande_status es = map_error(E, hs.error);
    if (es != HANDE_OK) return es;
    *n = nd;
    if (nd > cap) return HANDE_ERR_CAPACITY;
    if (nd == 0) return HANDE_OK;
    if (!keys || !pops) return HANDE_ERR_INVALID;
    const int W = E.KW;
    // keys transposed on the device into the other list buffer (free between
    // iterations), then one copy
    uint64_t* stage = E.P.key[cur ^ 1];
    E.ops.keys_to_aos(E, E.P.key[cur], stage, nd, E.P.cap, E.stream);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(keys, stage, (size_t)nd * W * 8, cudaMemcpyDeviceToHost, E.stream));
    CK(cudaMemcpyAsync(pops, E.P.pop[cur], nd * 8, cudaMemcpyDeviceToHost, E.stream));
    if (hdiag) CK(cudaMemcpyAsync(hdiag, E.P.hdiag[cur], nd * 8, cudaMemcpyDeviceToHost, E.stream));
    if (flags) {   // masked into the other list's flag buffer (free between iterations)
      uint8_t* fstage = E.P.flags[cur ^ 1];
      const int blocks = (int)std::min<int64_t>((nd + 255) / 256, 4096);
      k_core_flags<<<blocks, 256, 0, E.stream>>>(E.P.flags[cur], fstage, nd);
      CK(cudaGetLastError());
      CK(cudaMemcpyAsync(flags, fstage, nd, cudaMemcpyDeviceToHost, E.stream));
    }
    CK(cudaStreamSynchronize(E.stream));
    return HANDE_OK;
  });
}

hande_status hande_set_walkers(hande_ctx* ctx, const uint64_t* keys, const int64_t* pops, const double* hdiag,
                               int64_t n) {
  if (!ctx || n < 1 || !keys || !pops) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    const int W = E.KW;
    if (n > E.P.max_det) throw Fail{HANDE_ERR_CAPACITY, "more walkers than state_capacity"};
    // the keys go to the other list buffer (free between iterations), are
    // checked there and transposed into the list's layout
    const int cur = E.cur;
    uint64_t* stage = E.P.key[cur ^ 1];
    CK(cudaMemcpyAsync(stage, keys, (size_t)n * W * 8, cudaMemcpyHostToDevice, E.stream));
    CK(cudaMemsetAsync(E.check_word, 0, sizeof(unsigned), E.stream));
    E.ops.check_keys(E, stage, n, E.check_word, E.stream);
    CK(cudaGetLastError());
    unsigned bits = 0;
    CK(cudaMemcpyAsync(&bits, E.check_word, sizeof bits, cudaMemcpyDeviceToHost, E.stream));
    CK(cudaStreamSynchronize(E.stream));
    if (bits & 1u) throw Fail{HANDE_ERR_INVALID, "a key has bits beyond the spin orbitals"};
    if (bits & 2u) throw Fail{HANDE_ERR_INVALID, "a key has the wrong electron numbers"};
    if (bits & 4u) throw Fail{HANDE_ERR_INVALID, "keys must be strictly ascending"};
    if (!(bits & 8u)) throw Fail{HANDE_ERR_INVALID, "the reference determinant must be in the list"};
    E.ops.keys_to_soa(E, stage, E.P.key[cur], n, E.P.cap, E.stream);
    CK(cudaMemcpyAsync(E.P.pop[cur], pops, n * 8, cudaMemcpyHostToDevice, E.stream));
    CK(cudaMemsetAsync(E.P.flags[cur], 0, n, E.stream));
    if (E.host_iter == 0) {   // no previous iteration's counts to size the buckets with
      CK(cudaMemsetAsync((char*)E.P.st + offsetof(DevState, nspawn_prev), 0, 8, E.stream));
      CK(cudaMemsetAsync((char*)E.P.st + offsetof(DevState, nuniq_prev), 0, 8, E.stream));
      k_attempt_bound<<<(int)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, E.stream>>>(E.P.pop[cur], n, E.P.st);
      CK(cudaGetLastError());
    }
    CK(cudaMemcpyAsync((char*)E.P.st + offsetof(DevState, ndet) + 8 * cur, &n, 8, cudaMemcpyHostToDevice, E.stream));
    if (hdiag) CK(cudaMemcpyAsync(E.P.hdiag[cur], hdiag, n * 8, cudaMemcpyHostToDevice, E.stream));
    else E.ops.hdiag(E, cur, n, E.stream);
    CK(cudaGetLastError());
    // before the first iteration with semi_stoch_start == 0 the deterministic
    // space is chosen from the new list; later an active space is kept (its
    // matrix unchanged) and its members flagged in the new list, which must
    // hold all of them
    if (E.core_size > 0 && E.core_start == 0 && E.host_iter == 0) {
      E.core_active = false;
      E.P.ncore = 0;
      drop_graphs(E, 1);
      select_core(E);
    } else if (E.core_active && E.P.ncore > 0) {
      CK(cudaMemsetAsync(E.check_word, 0, sizeof(unsigned), E.stream));
      E.ops.core_mark(E, cur, E.check_word, E.stream);
      CK(cudaGetLastError());
      unsigned missing = 0;
      CK(cudaMemcpyAsync(&missing, E.check_word, sizeof missing, cudaMemcpyDeviceToHost, E.stream));
      CK(cudaStreamSynchronize(E.stream));
      if (missing) {
        E.core_active = false;
        E.P.ncore = 0;
        drop_graphs(E, 1);
        throw Fail{HANDE_ERR_INVALID,
                   "the list lacks a deterministic-space determinant (hande_set_state replaces the space)"};
      }
    }
    CK(cudaStreamSynchronize(E.stream));
    return HANDE_OK;
  });
}

hande_status hande_get_state(hande_ctx* ctx, hande_state* out, uint64_t* core_keys, int64_t core_cap) {
  if (!ctx || !out) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    hande_status es = map_error(E, read_error(E));
    if (es != HANDE_OK) return es;
    DevState hs;
    CK(cudaMemcpyAsync(&hs, E.P.st, sizeof hs, cudaMemcpyDeviceToHost, E.stream));
    CK(cudaStreamSynchronize(E.stream));
    std::memset(out, 0, sizeof *out);
    out->iter = hs.iter;
    out->shift = hs.shift;
    out->nw_ref = hs.nw_ref;
    out->vary = hs.vary;
    out->core_active = E.core_active ? 1 : 0;
    out->ncore = E.core_active ? E.P.ncore : 0;
    out->tau = E.P.tau;
    std::memcpy(&out->rmax, &hs.rmax_bits, 8);
    if (!core_keys || out->ncore == 0) return HANDE_OK;
    if (out->ncore > core_cap) return HANDE_ERR_CAPACITY;
    // the core keys transposed on the device into the other list buffer (free
    // between iterations), then one copy
    uint64_t* stage = E.P.key[E.cur ^ 1];
    E.ops.keys_to_aos(E, E.core_key, stage, out->ncore, out->ncore, E.stream);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(core_keys, stage, (size_t)out->ncore * E.KW * 8, cudaMemcpyDeviceToHost, E.stream));
    CK(cudaStreamSynchronize(E.stream));
    return HANDE_OK;
  });
}

hande_status hande_set_state(hande_ctx* ctx, const hande_state* in, const uint64_t* core_keys) {
  if (!ctx || !in) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    if (in->iter < 0 || (in->vary != 0 && in->vary != 1) || in->nw_ref < 0 || !std::isfinite(in->shift))
      throw Fail{HANDE_ERR_INVALID, "bad run state (iteration, shift, vary latch or reference population)"};
    if (in->vary == 1 && in->nw_ref == 0)
      throw Fail{HANDE_ERR_INVALID, "a varying shift needs a nonzero reference population"};
    if (!(in->tau > 0.0) || !std::isfinite(in->tau) || !(in->rmax >= 0.0) || !std::isfinite(in->rmax))
      throw Fail{HANDE_ERR_INVALID, "bad time step or time-step-search maximum"};
    const int64_t ncore = in->core_active ? in->ncore : 0;
    if (in->core_active && (E.core_size <= 0 || ncore < 1 || ncore > E.core_size || !core_keys))
      throw Fail{HANDE_ERR_INVALID, "deterministic space: needs semi_stoch_size >= ncore >= 1 and its keys"};
    const int cur = E.cur;
    const int64_t nd = read_i64(E, offsetof(DevState, ndet) + 8 * cur);
    if (ncore > nd) throw Fail{HANDE_ERR_INVALID, "deterministic space larger than the walker list"};
    if (ncore > 0) {
      // check the keys (ascending, electron numbers, the reference among them)
      // in the other list buffer, then transpose them into the core's layout
      uint64_t* stage = E.P.key[cur ^ 1];
      CK(cudaMemcpyAsync(stage, core_keys, (size_t)ncore * E.KW * 8, cudaMemcpyHostToDevice, E.stream));
      CK(cudaMemsetAsync(E.check_word, 0, sizeof(unsigned), E.stream));
      E.ops.check_keys(E, stage, ncore, E.check_word, E.stream);
      CK(cudaGetLastError());
      unsigned bits = 0;
      CK(cudaMemcpyAsync(&bits, E.check_word, sizeof bits, cudaMemcpyDeviceToHost, E.stream));
      CK(cudaStreamSynchronize(E.stream));
      if (bits & 7u) throw Fail{HANDE_ERR_INVALID, "core keys must be valid determinants in ascending order"};
      if (!(bits & 8u)) throw Fail{HANDE_ERR_INVALID, "the reference determinant must be in the core"};
      reserve_core(E, ncore);
      E.ops.keys_to_soa(E, stage, E.core_key, ncore, ncore, E.stream);
    }
    E.P.ncore = (int)ncore;
    E.P.core_key = E.core_key;
    CK(cudaMemsetAsync(E.check_word, 0, sizeof(unsigned), E.stream));
    E.ops.core_mark(E, cur, E.check_word, E.stream);
    CK(cudaGetLastError());
    unsigned missing = 0;
    CK(cudaMemcpyAsync(&missing, E.check_word, sizeof missing, cudaMemcpyDeviceToHost, E.stream));
    CK(cudaStreamSynchronize(E.stream));
    if (missing) {
      E.P.ncore = 0;
      E.core_active = false;
      drop_graphs(E, 1);
      throw Fail{HANDE_ERR_INVALID, "a deterministic-space determinant is not in the walker list"};
    }
    E.core_active = false;
    drop_graphs(E, 1);
    if (ncore > 0) build_core_tables(E);
    // counters of the run: iteration, shift, its latch and reference population
    DevState* st = E.P.st;
    CK(cudaMemcpyAsync((char*)st + offsetof(DevState, iter), &in->iter, 8, cudaMemcpyHostToDevice, E.stream));
    CK(cudaMemcpyAsync((char*)st + offsetof(DevState, shift), &in->shift, 8, cudaMemcpyHostToDevice, E.stream));
    CK(cudaMemcpyAsync((char*)st + offsetof(DevState, nw_ref), &in->nw_ref, 8, cudaMemcpyHostToDevice, E.stream));
    const int vary = in->vary;
    CK(cudaMemcpyAsync((char*)st + offsetof(DevState, vary), &vary, sizeof(int), cudaMemcpyHostToDevice, E.stream));
    unsigned long long rbits = 0;
    std::memcpy(&rbits, &in->rmax, 8);
    CK(cudaMemcpyAsync((char*)st + offsetof(DevState, rmax_bits), &rbits, 8, cudaMemcpyHostToDevice, E.stream));
    // the time step (and its spawn-weight factors) and the search state
    set_tau(E, in->tau, true);
    E.tau_searching = E.tau_search_on && !in->vary;
    E.P.tau_search = E.tau_searching ? 1 : 0;
    E.P.sys.want_r = E.P.tau_search;
    drop_graphs(E, 0);
    drop_graphs(E, 1);
    CK(cudaStreamSynchronize(E.stream));
    E.host_iter = in->iter;
    E.fetched = in->iter;
    return HANDE_OK;
  });
}

hande_status hande_set_proposal(hande_ctx* ctx, const uint32_t* q) {
  if (!ctx || !q) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    if (!E.ptab) throw Fail{HANDE_ERR_INVALID, "the context has no proposal table (UEG with excit_gen = 1)"};
    proposal_set(E, q);
    return HANDE_OK;
  });
}

hande_status hande_get_proposal(hande_ctx* ctx, uint32_t* q) {
  if (!ctx || !q) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    if (!E.ptab) throw Fail{HANDE_ERR_INVALID, "the context has no proposal table (UEG with excit_gen = 1)"};
    proposal_get(E, q);
    return HANDE_OK;
  });
}

hande_status hande_learn_proposal(hande_ctx* ctx, const hande_learning* learning) {
  if (!ctx || !learning) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    learner_attach(E, *learning);
    // the captured iterations now record training samples
    drop_graphs(E, 0);
    drop_graphs(E, 1);
    learner_refresh(E);
    return HANDE_OK;
  });
}

hande_status hande_learn_params(hande_ctx* ctx, float* get, const float* set, int64_t n, int64_t* n_out) {
  if (!ctx) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    if (!E.learn) throw Fail{HANDE_ERR_INVALID, "no learned proposal attached"};
    if (n_out) *n_out = learner_nparam(E);
    if (!get && !set) return HANDE_OK;
    if (n != learner_nparam(E)) throw Fail{HANDE_ERR_INVALID, "parameter count mismatch"};
    learner_params(E, get, set);
    return HANDE_OK;
  });
}

hande_status hande_learn_gradients(hande_ctx* ctx, const int32_t* rows, const int32_t* targets, const float* weights,
                                   int n, float* grads, double* loss) {
  if (!ctx || !rows || !targets || !weights || !grads || !loss) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    if (!E.learn) throw Fail{HANDE_ERR_INVALID, "no learned proposal attached"};
    learner_gradients(E, rows, targets, weights, n, grads, loss);
    return HANDE_OK;
  });
}

hande_status hande_learn_probabilities(hande_ctx* ctx, const int32_t* rows, int n, float* probs) {
  if (!ctx || !rows || !probs) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    if (!E.learn) throw Fail{HANDE_ERR_INVALID, "no learned proposal attached"};
    learner_probabilities(E, rows, n, probs);
    return HANDE_OK;
  });
}

hande_status hande_learn_refresh(hande_ctx* ctx) {
  if (!ctx) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    if (!E.learn) throw Fail{HANDE_ERR_INVALID, "no learned proposal attached"};
    learner_refresh(E);
    return HANDE_OK;
  });
}

hande_status hande_autotune(hande_ctx* ctx, int iterations, hande_tuning* out) {
  if (!ctx || iterations < 1) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  if (E.failed) return HANDE_ERR_STATE;
  return run_guarded(&E, [&]() -> hande_status {
    const int dflt_sp = E.P.bucket_spawns, dflt_new = E.P.bucket_new, dflt_grid = E.attempt_grid;
    int nsm = 0;
    CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, E.device));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    struct Cleanup {
      cudaEvent_t a, b;
      ~Cleanup() {
        cudaEventDestroy(a);
        cudaEventDestroy(b);
      }
    } cleanup{e0, e1};
    hande_tuning best{dflt_sp, dflt_new, dflt_grid, -1.0};
    for (double fs : {0.5, 0.75, 1.0, 1.25})
      for (double fn : {0.5, 1.0})
        for (int per_sm : {1, 2}) {
          const int grid = std::min(dflt_grid, per_sm * nsm);
          E.P.bucket_spawns = std::max(1, (int)(dflt_sp * fs));
          E.P.bucket_new = dflt_new > 0 ? std::max(1, (int)(dflt_new * fn)) : 0;
          E.attempt_grid = grid;
          drop_graphs(E, 0);
          drop_graphs(E, 1);
          hande_status st = hande_iterate(ctx, 1);   // captures the graphs for this shape
          if (st == HANDE_OK && iterations >= kGraphIters)
            for (int c = 0; c < 2; ++c) ensure_graph(E, c, E.core_active ? 1 : 0, kGraphIters);
          if (st == HANDE_OK) {
            CK(cudaEventRecord(e0, E.stream));
            st = hande_iterate(ctx, iterations);
          }
          if (st != HANDE_OK) {   // back to the defaults (the context may still be usable)
            E.P.bucket_spawns = dflt_sp;
            E.P.bucket_new = dflt_new;
            E.attempt_grid = dflt_grid;
            drop_graphs(E, 0);
            drop_graphs(E, 1);
            return st;
          }
          CK(cudaEventRecord(e1, E.stream));
          CK(cudaEventSynchronize(e1));
          float ms = 0.0f;
          CK(cudaEventElapsedTime(&ms, e0, e1));
          const double per = ms / iterations;
          if (best.ms_per_iteration < 0.0 || per < best.ms_per_iteration)
            best = hande_tuning{E.P.bucket_spawns, E.P.bucket_new, grid, per};
        }
    E.P.bucket_spawns = best.bucket_spawns;
    E.P.bucket_new = best.bucket_new;
    E.attempt_grid = best.attempt_blocks;
    drop_graphs(E, 0);
    drop_graphs(E, 1);
    if (out) *out = best;
    return map_error(E, read_error(E));
  });
}

hande_status hande_diagnostics(hande_ctx* ctx, hande_diag* out) {
  if (!ctx || !out) return HANDE_ERR_INVALID;
  Engine& E = ctx->E;
  return run_guarded(&E, [&]() -> hande_status {
    DevState hs;
    CK(cudaMemcpyAsync(&hs, E.P.st, sizeof hs, cudaMemcpyDeviceToHost, E.stream));
    CK(cudaStreamSynchronize(E.stream));
    std::memset(out, 0, sizeof *out);
    out->error_bits = hs.error | E.err_bits;
    out->ndet = hs.ndet[E.cur];
    out->natt = hs.natt;
    out->nspawn = hs.nspawn;
    out->nbuckets = hs.nbuckets;
    out->bucket_main = hs.sb;
    out->tile_capacity = E.P.tile_cap;
    out->ncore = E.P.ncore;
    // det pass, attempts, then match, decide, place, write; or split, buckets, bucket scan, scatter, annihilation (1, or 5 on the warp
    // path), new diagonals, finalize; and the deterministic-space projection (3)
    // once it is active
    out->launches_per_iteration = (E.P.hash_merge ? 6 : 9 + (E.merge_warp ? 4 : 0)) +
                                  (E.core_active && E.P.ncore > 0 ? 3 : 0);
    out->deferred_buckets = hs.ndefer + hs.nbig;
    int64_t nb = std::min<int64_t>(hs.nbuckets, E.P.cap);
    if (nb > 0) {
      std::vector<uint32_t> cnt((size_t)nb);
      CK(cudaMemcpyAsync(cnt.data(), E.P.hash_merge ? E.P.g_new : E.P.bcount, nb * 4, cudaMemcpyDeviceToHost, E.stream));
      CK(cudaStreamSynchronize(E.stream));
      for (uint32_t c : cnt) out->max_bucket_spawns = std::max<int64_t>(out->max_bucket_spawns, c);
    }
    return HANDE_OK;
  });
}

hande_status hande_reference(hande_ctx* ctx, double* e_ref, uint64_t* key) {
  if (!ctx) return HANDE_ERR_INVALID;
  if (e_ref) *e_ref = ctx->E.e_ref;
  if (key)
    for (int j = 0; j < ctx->E.KW; ++j) key[j] = ctx->E.P.d0[j];
  return HANDE_OK;
}

int64_t hande_iterations(const hande_ctx* ctx) { return ctx ? ctx->E.host_iter : 0; }

void hande_destroy(hande_ctx* ctx) {
  if (!ctx) return;
  release_all(ctx->E);
  delete ctx;
}

const char* hande_last_error(const hande_ctx* ctx) {
  if (!ctx) return "no context";
  return ctx->E.err.c_str();
}

}  // extern "C"
