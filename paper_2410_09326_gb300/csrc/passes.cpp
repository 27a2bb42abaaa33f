// Host passes: virtual swap, k-qubit fusion and block classification.
//
// Virtual swap (Sec. III-D): a SWAP gate exchanges two qubits' roles; instead
// of moving 2^(n-1) amplitudes, the pass swaps the two entries of the
// logical->physical map and later gates are renamed through it.
//
// Fusion generalises single-qubit gate merging (Sec. III-D, Z-Y
// decomposition: consecutive one-qubit gates collapse into one unitary) and
// QCOR's two-qubit block merging (Sec. IV, "all-on" set) to blocks of up to k
// qubits whose product matrix is formed in FP64 on the host.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <thread>

#include "qs_internal.h"

namespace qs {

namespace {

constexpr double kEps = 1e-14;

bool is_one(cd z) { return std::norm(z - cd(1, 0)) <= kEps * kEps; }
bool is_zero(cd z) { return std::norm(z) <= kEps * kEps; }

int popcount64(uint64_t x) { return __builtin_popcountll(x); }

// Position of physical qubit q inside the sorted list qs[0..w).
int pos_of(const int *qs, int w, int q) {
  for (int i = 0; i < w; i++)
    if (qs[i] == q) return i;
  return -1;
}

// A block's product under construction: 2^w x 2^w, real and imaginary parts
// apart, so that the loops over a row's columns vectorise.
struct Product {
  int d;
  std::vector<double> re, im, tre, tim;
  explicit Product(int w) : d(1 << w), re((size_t)d * d, 0.0), im((size_t)d * d, 0.0), tre(8 * d), tim(8 * d) {
    for (int i = 0; i < d; i++) re[(size_t)i * d + i] = 1;
  }
  cd at(int r, int c) const { return cd(re[(size_t)r * d + c], im[(size_t)r * d + c]); }
};

// Applies a gate's full matrix G (on local positions pos[0..m), m <= 3) from
// the left: row combinations, zero entries and unchanged rows skipped.
void left_multiply(Product &M, const std::vector<cd> &G, const int *pos, int m) {
  const int d = M.d, dg = 1 << m;
  int gmask = 0, off[8];
  for (int j = 0; j < m; j++) gmask |= 1 << pos[j];
  bool same[8];
  for (int l = 0; l < dg; l++) {
    off[l] = 0;
    for (int j = 0; j < m; j++)
      if ((l >> j) & 1) off[l] |= 1 << pos[j];
    same[l] = true;
    for (int b = 0; b < dg; b++) same[l] = same[l] && G[(size_t)l * dg + b] == cd(b == l ? 1 : 0, 0);
  }
  for (int base = 0; base < d; base++) {
    if (base & gmask) continue;
    for (int a = 0; a < dg; a++) {
      if (same[a]) continue;
      double *tr = M.tre.data() + (size_t)a * d, *ti = M.tim.data() + (size_t)a * d;
      bool first = true;
      for (int b = 0; b < dg; b++) {
        const double gr = G[(size_t)a * dg + b].real(), gi = G[(size_t)a * dg + b].imag();
        if (gr == 0 && gi == 0) continue;
        const double *xr = M.re.data() + (size_t)(base | off[b]) * d, *xi = M.im.data() + (size_t)(base | off[b]) * d;
        if (first)
          for (int c = 0; c < d; c++) {
            tr[c] = gr * xr[c] - gi * xi[c];
            ti[c] = gr * xi[c] + gi * xr[c];
          }
        else
          for (int c = 0; c < d; c++) {
            tr[c] += gr * xr[c] - gi * xi[c];
            ti[c] += gr * xi[c] + gi * xr[c];
          }
        first = false;
      }
    }
    for (int a = 0; a < dg; a++) {
      if (same[a]) continue;
      std::memcpy(M.re.data() + (size_t)(base | off[a]) * d, M.tre.data() + (size_t)a * d, sizeof(double) * d);
      std::memcpy(M.im.data() + (size_t)(base | off[a]) * d, M.tim.data() + (size_t)a * d, sizeof(double) * d);
    }
  }
}

// Runs f(0..n) on as many host threads (up to 16) as work_us, the estimated
// microseconds of all the calls together, pays for: starting and joining a
// thread costs about as much as 50 us of work, so a thread is given 100.
template <typename F> void parallel_for(size_t n, double work_us, F f) {
  const unsigned most = std::min(16u, std::max(1u, std::thread::hardware_concurrency()));
  const size_t nt = std::min<size_t>({most, n, (size_t)(work_us / 100) + 1});
  if (nt <= 1) {
    for (size_t i = 0; i < n; i++) f(i);
    return;
  }
  std::atomic<size_t> next{0};
  auto work = [&] {
    for (size_t i; (i = next.fetch_add(1)) < n;) f(i);
  };
  std::vector<std::thread> th;
  th.reserve(nt - 1);
  for (size_t t = 1; t < nt; t++) th.emplace_back(work);
  work();
  for (auto &x : th) x.join();
}

// As many gates of a long list as these cost roll-outs of `horizon` gates: a
// short list's roll-outs end with it, and have fewer blocks to try.
double roll_out_gates(size_t gates, int horizon) {
  return (double)gates * std::min(1.0, (double)gates / (2.0 * (double)std::max(horizon, 1)));
}

struct Pending {
  std::vector<int> members;  // indices into the physical gate list
  uint64_t qmask = 0;
  bool all_diag = true;
  uint64_t tmask = 0;       // qubits some member acts on non-diagonally
  uint64_t out_union = 0;   // tile sub-groups: member qubits outside the tile
  uint64_t cl_and = ~0ull;  // tile sub-groups: qubits every member is the identity on when 0
};

// Commuting greedy grouping of the gates pg[idx[..]] (ascending list order):
// a gate may join any group at or after the last group it cannot commute
// past (two gates commute when both act diagonally on every qubit they
// share); it joins the first such group `fits` accepts, else a new one.
struct NoJoin {
  void operator()(Pending &, int, uint64_t) const {}
};

template <typename Fits, typename Joined = NoJoin>
void greedy_groups(const std::vector<qs_gate> &pg, const std::vector<int> &idx, std::vector<Pending> &groups,
                   Fits fits, Joined joined = Joined()) {
  std::vector<int> last_any(64, -1), last_nd(64, -1);
  for (int i : idx) {
    const qs_gate &g = pg[i];
    uint64_t gmask = 0, gt = 0;
    int lower = -1;
    for (int j = 0; j < g.nq; j++) {
      const int q = g.q[j];
      gmask |= 1ull << q;
      if (!gate_diag_on(g, j)) gt |= 1ull << q;
      lower = std::max(lower, gate_diag_on(g, j) ? last_nd[q] : last_any[q]);
    }
    const bool gdiag = op_info(g.op).diagonal;
    int chosen = -1;
    for (int b = std::max(lower, 0); b < (int)groups.size(); b++)
      if (fits(groups[b], i, gmask, gt, gdiag)) {
        chosen = b;
        break;
      }
    if (chosen < 0) {
      groups.emplace_back();
      chosen = (int)groups.size() - 1;
    }
    Pending &p = groups[chosen];
    p.members.push_back(i);
    p.qmask |= gmask;
    p.tmask |= gt;
    p.all_diag = p.all_diag && gdiag;
    joined(p, i, gmask);
    for (int j = 0; j < g.nq; j++) {
      const int q = g.q[j];
      last_any[q] = std::max(last_any[q], chosen);
      if (!gate_diag_on(g, j)) last_nd[q] = std::max(last_nd[q], chosen);
    }
  }
}

// Fusion with a roll-out look-ahead (a pilot method): where a gate could join
// several blocks (the first four that fit) or open a new one, each choice is
// followed by `horizon` gates of plain first-fit placement, and the choice
// whose roll-out ends with the fewest blocks -- then the narrowest recent
// blocks -- is kept; ties keep the earliest candidate (first fit). Placement
// obeys the same commutation rule as greedy_groups, and the limits that
// fits(group, gate) states. With free_joins a gate whose first candidate needs
// no further qubit for it joins that one without roll-outs: it widens nothing
// and holds later gates back the least.
struct LookGroup {
  uint64_t qmask, tmask;  // its qubits; those some member acts on non-diagonally
  bool all_diag;
};

template <typename Fits>
void lookahead_groups(const std::vector<qs_gate> &pg, const std::vector<int> &idx, std::vector<Pending> &groups,
                      Fits fits_gate, int horizon, int tail_blocks, bool free_joins) {
  using LG = LookGroup;
  struct GI {
    uint64_t gmask, gt;
    bool gdiag;
    int nq;
    int q[6];
    bool dq[6];
  };
  const int N = (int)idx.size();
  std::vector<GI> info(N);
  for (int i = 0; i < N; i++) {
    const qs_gate &g = pg[idx[i]];
    GI &x = info[i];
    x.gmask = x.gt = 0;
    x.gdiag = op_info(g.op).diagonal;
    x.nq = g.nq;
    for (int j = 0; j < g.nq; j++) {
      x.q[j] = g.q[j];
      x.dq[j] = gate_diag_on(g, j);
      x.gmask |= 1ull << g.q[j];
      if (!x.dq[j]) x.gt |= 1ull << g.q[j];
    }
  }
  auto lower_of = [](const GI &x, const int *la, const int *ln) {
    int lower = -1;
    for (int j = 0; j < x.nq; j++) lower = std::max(lower, x.dq[j] ? ln[x.q[j]] : la[x.q[j]]);
    return lower;
  };
  auto fits = [&](const LG &b, const GI &x) { return fits_gate(b, LG{x.gmask, x.gt, x.gdiag}); };
  auto place = [](std::vector<LG> &G, int *la, int *ln, const GI &x, int ch) {
    if (ch == (int)G.size()) G.push_back({0, 0, true});
    G[ch].qmask |= x.gmask;
    G[ch].tmask |= x.gt;
    G[ch].all_diag = G[ch].all_diag && x.gdiag;
    for (int j = 0; j < x.nq; j++) {
      la[x.q[j]] = std::max(la[x.q[j]], ch);
      if (!x.dq[j]) ln[x.q[j]] = std::max(ln[x.q[j]], ch);
    }
  };
  std::vector<LG> G, G2;
  int la[64], ln[64], la2[64], ln2[64];
  for (int q = 0; q < 64; q++) la[q] = ln[q] = -1;
  for (int i = 0; i < N; i++) {
    const GI &x = info[i];
    const int lower = std::max(lower_of(x, la, ln), 0);
    int cand[5], nc = 0;
    for (int b = lower; b < (int)G.size() && nc < 4; b++)
      if (fits(G[b], x)) cand[nc++] = b;
    cand[nc++] = (int)G.size();
    int ch = cand[0];
    const bool join = free_joins && nc > 1 && (x.gmask & ~G[ch].qmask) == 0 && (x.gdiag || !G[ch].all_diag);
    if (nc > 1 && horizon > 0 && !join) {
      long best_blocks = -1, best_tail = 0;
      for (int c = 0; c < nc; c++) {
        G2 = G;
        std::memcpy(la2, la, sizeof(la));
        std::memcpy(ln2, ln, sizeof(ln));
        place(G2, la2, ln2, x, cand[c]);
        const int end = std::min(N, i + 1 + horizon);
        // (the block count only grows: a roll-out past the best one's is lost)
        for (int j = i + 1; j < end && (best_blocks < 0 || (long)G2.size() <= best_blocks); j++) {
          const GI &y = info[j];
          int b = std::max(lower_of(y, la2, ln2), 0);
          while (b < (int)G2.size() && !fits(G2[b], y)) b++;
          place(G2, la2, ln2, y, b);
        }
        long tail = 0;
        for (int b = std::max(0, (int)G2.size() - tail_blocks); b < (int)G2.size(); b++)
          tail += popcount64(G2[b].qmask);
        if (best_blocks < 0 || (long)G2.size() < best_blocks ||
            ((long)G2.size() == best_blocks && tail < best_tail)) {
          best_blocks = (long)G2.size();
          best_tail = tail;
          ch = cand[c];
        }
      }
    }
    place(G, la, ln, x, ch);
    if (ch == (int)groups.size()) groups.emplace_back();
    Pending &p = groups[ch];
    p.members.push_back(idx[i]);
    p.qmask |= x.gmask;
    p.tmask |= x.gt;
    p.all_diag = p.all_diag && x.gdiag;
  }
}

// Qubits on which the gate is the identity whenever that qubit is 0 (the
// controls of a controlled gate; both qubits of CZ / CPhase; the qubit of a
// phase gate diag(1, e^{ia})). A block made only of such gates on a qubit has
// that qubit as a detected control.
uint64_t ctrl_like_mask(const qs_gate &g) {
  const OpInfo &oi = op_info(g.op);
  uint64_t m = 0;
  if (!oi.diagonal) {
    for (int j = 0; j < oi.nctrl; j++) m |= 1ull << g.q[j];
    return m;
  }
  std::vector<cd> G;
  gate_full_matrix(g, G);
  const int d = 1 << g.nq;
  for (int j = 0; j < g.nq; j++) {
    bool ok = true;
    for (int l = 0; l < d && ok; l++)
      if (!((l >> j) & 1) && !is_one(G[(size_t)l * d + l])) ok = false;
    if (ok) m |= 1ull << g.q[j];
  }
  return m;
}

// Turns a group of gates into a classified Block (dense/diag/permute);
// returns false when the product is the identity (nothing to launch).
double wrap_angle(double a) {
  a = std::remainder(a, 2 * M_PI);  // [-pi, pi]
  return a <= -M_PI ? a + 2 * M_PI : a;
}

// Phase polynomial of a run of diagonal gates (each on at most two qubits):
// gate g contributes arg g(00) + (arg g(10) - arg g(00)) x_0 +
// (arg g(01) - arg g(00)) x_1 + (arg g(11) - arg g(10) - arg g(01) +
// arg g(00)) x_0 x_1, which equals arg g(x) on all four inputs. Returns false
// when the product is the identity.
bool phase_block(const std::vector<qs_gate> &pg, const Pending &p, const int *qs, int w, Block &out) {
  std::vector<double> a(w, 0.0), b((size_t)w * (w - 1) / 2, 0.0);
  double c = 0;
  std::vector<cd> G;
  for (int gi : p.members) {
    const qs_gate &g = pg[gi];
    gate_full_matrix(g, G);
    const int d = 1 << g.nq;
    double ph[4] = {0, 0, 0, 0};
    for (int l = 0; l < d; l++) ph[l] = std::arg(G[(size_t)l * d + l]);
    const int j0 = pos_of(qs, w, g.q[0]);
    c += ph[0];
    a[j0] += ph[1] - ph[0];
    if (g.nq == 2) {
      const int j1 = pos_of(qs, w, g.q[1]);
      a[j1] += ph[2] - ph[0];
      const double x = ph[3] - ph[1] - ph[2] + ph[0];
      b[j0 < j1 ? tri_index(j0, j1, w) : tri_index(j1, j0, w)] += x;
    }
  }
  // keep the qubits that still carry a term
  auto zero = [](double v) { return std::fabs(wrap_angle(v)) <= kEps; };
  std::vector<char> used(w, 0);
  for (int j = 0; j < w; j++) {
    if (!zero(a[j])) used[j] = 1;
    for (int l = j + 1; l < w; l++)
      if (!zero(b[tri_index(j, l, w)])) used[j] = used[l] = 1;
  }
  std::vector<int> keep;
  for (int j = 0; j < w; j++)
    if (used[j]) keep.push_back(j);
  const int k = (int)keep.size();
  if (k == 0 && zero(c)) return false;
  out.kind = BK_PHASE;
  out.k = k;
  out.ph_c = wrap_angle(c);
  out.ph_q.resize(k);
  out.ph_a.resize(k);
  out.ph_b.assign(k > 1 ? (size_t)k * (k - 1) / 2 : 0, 0.0);
  for (int j = 0; j < k; j++) {
    out.ph_q[j] = qs[keep[j]];
    out.ph_a[j] = wrap_angle(a[keep[j]]);
    for (int l = j + 1; l < k; l++) out.ph_b[tri_index(j, l, k)] = wrap_angle(b[tri_index(keep[j], keep[l], w)]);
  }
  for (int j = 0; j < std::min(k, QS_MAX_DIAG); j++) out.q[j] = out.ph_q[j];
  return true;
}

// table_max: widest diagonal run kept as a phase table; wider all-diagonal
// groups become phase polynomials when phase_ok.
bool finish_block(const std::vector<qs_gate> &pg, const Pending &p, bool allow_permute, Block &out,
                  int table_max = QS_MAX_DIAG, bool phase_ok = false) {
  int qs[64], w = 0;
  for (int q = 0; q < 64; q++)
    if ((p.qmask >> q) & 1) qs[w++] = q;
  out = Block();
  out.n_gates = (int)p.members.size();
  const qs_gate &g0 = pg[p.members[0]];
  if (out.n_gates == 1) {
    out.first_op = g0.op;
    out.meta = g0.op == QS_SWAP ? 3 : (op_info(g0.op).nq == 1 ? 0 : 1);
  }
  if (allow_permute && out.n_gates == 1 && g0.op == QS_SWAP) {
    out.kind = BK_PERMUTE;
    out.k = 2;
    out.q[0] = std::min(g0.q[0], g0.q[1]);
    out.q[1] = std::max(g0.q[0], g0.q[1]);
    return true;
  }
  std::vector<cd> G;
  if (p.all_diag && phase_ok && w > table_max) {
    const int first_op = out.first_op, meta = out.meta, ng = out.n_gates;
    if (!phase_block(pg, p, qs, w, out)) return false;
    out.first_op = first_op;
    out.meta = meta;
    out.n_gates = ng;
    return true;
  }
  if (p.all_diag) {
    // diagonal table over the w qubits: product of every member's diagonal
    std::vector<cd> tab((size_t)1 << w, cd(1, 0));
    for (int gi : p.members) {
      const qs_gate &g = pg[gi];
      gate_full_matrix(g, G);
      int m = g.nq, dg = 1 << m;
      int pos[8];
      for (int j = 0; j < m; j++) pos[j] = pos_of(qs, w, g.q[j]);
      for (size_t l = 0; l < tab.size(); l++) {
        int lg = 0;
        for (int j = 0; j < m; j++) lg |= (int)((l >> pos[j]) & 1) << j;
        tab[l] *= G[(size_t)lg * dg + lg];
      }
    }
    // a qubit whose 0 half carries phase 1 everywhere acts as a control
    uint64_t cmask = 0;
    int keep[64], nk = 0;
    for (int j = 0; j < w; j++) {
      bool ctrl = true;
      for (size_t l = 0; l < tab.size() && ctrl; l++)
        if (!((l >> j) & 1) && !is_one(tab[l])) ctrl = false;
      if (ctrl) cmask |= 1ull << qs[j];
      else keep[nk++] = j;
    }
    int cbits = 0;
    for (int j = 0; j < w; j++)
      if ((cmask >> qs[j]) & 1) cbits |= 1 << j;
    std::vector<cd> t2((size_t)1 << nk);
    bool identity = true;
    for (size_t l2 = 0; l2 < t2.size(); l2++) {
      int l = cbits;
      for (int j = 0; j < nk; j++)
        if ((l2 >> j) & 1) l |= 1 << keep[j];
      t2[l2] = tab[l];
      if (!is_one(t2[l2])) identity = false;
    }
    if (identity) return false;
    out.kind = BK_DIAG;
    out.k = nk;
    for (int j = 0; j < nk; j++) out.q[j] = qs[keep[j]];
    out.cmask = cmask;
    out.nctrl = popcount64(cmask);
    out.mat = std::move(t2);
    return true;
  }
  // dense product over the w qubits
  const int d = 1 << w;
  Product M(w);
  for (int gi : p.members) {
    const qs_gate &g = pg[gi];
    gate_full_matrix(g, G);
    int pos[8];
    for (int j = 0; j < g.nq; j++) pos[j] = pos_of(qs, w, g.q[j]);
    left_multiply(M, G, pos, g.nq);
  }
  // control detection: block-diagonal in bit j with identity on the 0 half
  uint64_t cmask = 0;
  int keep[64], nk = 0;
  for (int j = 0; j < w; j++) {
    bool ctrl = true;
    for (int r = 0; r < d && ctrl; r++)
      for (int c = 0; c < d && ctrl; c++) {
        cd z = M.at(r, c);
        int br = (r >> j) & 1, bc = (c >> j) & 1;
        if (br != bc) { if (!is_zero(z)) ctrl = false; }
        else if (br == 0) { if (r == c ? !is_one(z) : !is_zero(z)) ctrl = false; }
      }
    if (ctrl) cmask |= 1ull << qs[j];
    else keep[nk++] = j;
  }
  int cbits = 0;
  for (int j = 0; j < w; j++)
    if ((cmask >> qs[j]) & 1) cbits |= 1 << j;
  const int dk = 1 << nk;
  std::vector<cd> R((size_t)dk * dk);
  bool diag = true, identity = true;
  auto expand = [&](int l2) {
    int l = cbits;
    for (int j = 0; j < nk; j++)
      if ((l2 >> j) & 1) l |= 1 << keep[j];
    return l;
  };
  for (int r = 0; r < dk; r++) {
    const int er = expand(r);
    for (int c = 0; c < dk; c++) {
      cd z = M.at(er, nk == w ? c : expand(c));
      R[(size_t)r * dk + c] = z;
      if (diag && r != c && !is_zero(z)) diag = false, identity = false;
      if (identity && r == c && !is_one(z)) identity = false;
    }
  }
  if (identity) return false;
  out.cmask = cmask;
  out.nctrl = popcount64(cmask);
  out.k = nk;
  for (int j = 0; j < nk; j++) out.q[j] = qs[keep[j]];
  if (diag && nk <= QS_MAX_DIAG) {
    out.kind = BK_DIAG;
    out.mat.resize(dk);
    for (int i = 0; i < dk; i++) out.mat[i] = R[(size_t)i * dk + i];
  } else {
    out.kind = BK_DENSE;
    out.mat = std::move(R);
  }
  return true;
}

// Estimated host time of the groups' products: a gate on a w-qubit dense
// block updates 4^w entries at about a nanosecond each, on a diagonal one 2^w.
double products_us(const std::vector<Pending> &groups) {
  double us = 0;
  for (const Pending &p : groups) {
    const int w = popcount64(p.qmask);
    us += 0.3 + (double)p.members.size() * (0.1 + 1e-3 * (p.all_diag ? (w <= QS_MAX_DIAG ? 4.0 * (1 << w) : 100.0)
                                                                     : std::ldexp(1.0, 2 * w)));
  }
  return us;
}

void push_exchanges(const std::vector<std::pair<int, int>> &reloc, std::vector<Block> &plan) {
  for (auto &pr : reloc) {  // the exchanges run first
    Block b;
    b.kind = BK_PERMUTE;
    b.k = 2;
    b.q[0] = std::min(pr.first, pr.second);
    b.q[1] = std::max(pr.first, pr.second);
    b.n_gates = 0;
    b.meta = 3;
    plan.push_back(std::move(b));
  }
}

constexpr int kSearchBits = 23;      // narrowest complex64 state whose fusion is searched
constexpr int kFullSearchBits = 27;  // and without free joins too

constexpr int kTileMaxOps = 64;     // member blocks of one tile pass
constexpr int kTilePool = 2048;     // matrix + phase-table entries of one tile pass

// Cache-blocked passes (the GPU analogue of the chunk segment that virtual
// swap keeps hot qubits in, Sec. III-D): gates are grouped, with the same
// commutation rule as fusion, into passes whose non-diagonal qubits fit one
// tile of m qubits that always contains bits 0..kTileLowBits-1. A pass then
// costs one HBM read and write: each CTA loads a tile of 2^m amplitudes
// into shared memory, applies the pass's member blocks there, and stores it.
// Inside a pass the gates are fused again, at most tile_k qubits wide; a
// qubit outside the tile may only be a control or sit in a diagonal block.
// repeated (batches): a pass with one member stays a pass, and diagonal runs
// become phase polynomials of any width.
qs_status tile_plan(int n, const std::vector<qs_gate> &pg, const std::vector<int> &all, const qs_opts &opts,
                    bool c128, bool repeated, std::vector<Block> &out, std::string &err) {
  const int m = tile_bits_of(opts, c128);
  const int kin = tile_k_of(opts);
  const int D = std::max(1, std::min(opts.diag_max, QS_MAX_DIAG));
  const uint64_t low = (1ull << kTileLowBits) - 1;
  std::vector<Pending> passes;
  greedy_groups(pg, all, passes, [&](const Pending &p, int, uint64_t, uint64_t gt, bool) {
    return popcount64(p.tmask | low | gt) <= m;
  });
  // tile qubits of every pass: its non-diagonal qubits, padded with the
  // lowest free bits (longer contiguous runs per load)
  std::vector<uint64_t> tmask(passes.size());
  for (size_t pi = 0; pi < passes.size(); pi++) {
    uint64_t t = passes[pi].tmask | low;
    for (int q = 0; q < n && popcount64(t) < m; q++) t |= 1ull << q;
    tmask[pi] = t;
  }
  std::vector<uint64_t> cl(pg.size(), 0);
  parallel_for(pg.size(), repeated ? 0 : 0.1 * (double)pg.size(), [&](size_t i) { cl[i] = ctrl_like_mask(pg[i]); });
  // member blocks of every pass
  std::vector<Pending> subs;
  std::vector<int> sub_pass;
  for (size_t pi = 0; pi < passes.size(); pi++) {
    const uint64_t T = tmask[pi];
    std::vector<Pending> sg;
    greedy_groups(
        pg, passes[pi].members, sg,
        [&](const Pending &p, int i, uint64_t gmask, uint64_t, bool gdiag) {
          const int width = popcount64(p.qmask | gmask);
          if (p.all_diag && gdiag) return repeated || width <= D;
          // a non-diagonal block may reach outside the tile only through
          // qubits that are controls of every member: then they are
          // detected as controls of the product
          const uint64_t out = p.out_union | (gmask & ~T);
          return width <= kin && (out & ~(p.cl_and & cl[i])) == 0;
        },
        [&](Pending &p, int i, uint64_t gmask) {
          p.out_union |= gmask & ~T;
          p.cl_and &= cl[i];
        });
    for (Pending &p : sg) {
      subs.push_back(std::move(p));
      sub_pass.push_back((int)pi);
    }
  }
  std::vector<Block> done(subs.size());
  std::vector<char> keep(subs.size(), 0);
  parallel_for(subs.size(), repeated ? 0 : products_us(subs), [&](size_t i) {
    keep[i] = finish_block(pg, subs[i], false, done[i], repeated ? 0 : QS_MAX_DIAG, repeated) ? 1 : 0;
  });
  (void)err;
  size_t si = 0;
  for (size_t pi = 0; pi < passes.size(); pi++) {
    const uint64_t T = tmask[pi];
    std::vector<Block> members;
    for (; si < subs.size() && sub_pass[si] == (int)pi; si++)
      if (keep[si]) members.push_back(std::move(done[si]));
    bool ok = true;
    for (const Block &b : members) {
      if (b.kind == BK_DENSE) {
        ok = ok && b.k <= 4;
        for (int j = 0; j < b.k; j++) ok = ok && ((T >> b.q[j]) & 1);
      } else if (b.kind == BK_DIAG) {
        for (int j = 0; j < b.k && repeated; j++) ok = ok && ((T >> b.q[j]) & 1);
      } else if (b.kind != BK_PHASE) {
        ok = false;
      }
    }
    if (!ok && repeated) {
      err = "tile pass with a member outside its tile";
      return QS_EUNSUPPORTED;
    }
    if (!ok) {  // cannot happen by construction; the members stay valid alone
      for (Block &b : members) out.push_back(std::move(b));
      continue;
    }
    // split at the shared-memory limits of one pass
    size_t b0 = 0;
    while (b0 < members.size()) {
      size_t b1 = b0;
      int pool = 0;
      while (b1 < members.size() && (int)(b1 - b0) < kTileMaxOps) {
        const Block &b = members[b1];
        const int ent = b.kind == BK_DENSE ? (1 << (2 * b.k)) : (b.kind == BK_PHASE ? (n + 4) * (n + 2) / 2 : 1 << b.k);
        if (b1 > b0 && pool + ent > kTilePool) break;
        pool += ent;
        b1++;
      }
      if (b1 - b0 == 1 && !repeated) {
        out.push_back(std::move(members[b0]));
      } else {
        Block t;
        t.kind = BK_TILE;
        t.k = m;
        int w = 0;
        for (int q = 0; q < 64; q++)
          if ((T >> q) & 1) t.tile_q[w++] = q;
        t.meta = 5;
        t.n_gates = 0;
        for (size_t j = b0; j < b1; j++) {
          t.n_gates += members[j].n_gates;
          t.sub.push_back(std::move(members[j]));
        }
        out.push_back(std::move(t));
      }
      b0 = b1;
    }
  }
  return QS_OK;
}

// Cost of a tile pass of b blocks, in launches of a single block of up to five
// targets: 0.45 + 0.4 b, fitted to passes at 27 qubits, where a block is an HBM
// pass, and as good at 19 qubits, where launches and latency count. (It puts
// the 39 passes of the 30-qubit random circuit, 116 blocks, at 64; they take
// 165 ms, the circuit's 126 blocks one by one 339.)
double tc_tile_cost(size_t b) { return 0.45 + 0.4 * (double)b; }

// Tensor-core tile passes (tc_tile.cu): gates grouped as in tile_plan into
// passes whose non-diagonal qubits fit a tile of kTcTileBits, each pass's gates into
// blocks of at most five qubits inside the tile and kTcTileSel outside it
// (there they act diagonally: the bits pick the matrix).
struct TcPass {
  uint64_t tile = 0;
  bool single = false;  // its blocks run one by one
  std::vector<Pending> blocks;
};

// The gates with every one-qubit gate moved back to just before the next gate
// on its qubit that has others, with which it then shares a block: first fit
// would take a layer's one-qubit gates in the order they come. 82 -> 77 blocks
// for a 19-qubit 30-layer random circuit.
std::vector<int> one_qubit_late(const std::vector<qs_gate> &pg, const std::vector<int> &idx) {
  std::vector<int> out, wait[64];
  out.reserve(idx.size());
  auto flush = [&](int q) {
    out.insert(out.end(), wait[q].begin(), wait[q].end());
    wait[q].clear();
  };
  for (int i : idx) {
    const qs_gate &g = pg[i];
    if (g.nq == 1) {
      wait[g.q[0]].push_back(i);
      continue;
    }
    for (int j = 0; j < g.nq; j++) flush(g.q[j]);
    out.push_back(i);
  }
  for (int q = 0; q < 64; q++) flush(q);
  return out;
}

// A pass whose gates cost less as blocks of K qubits one by one stays that, as
// does one that has no block of four qubits: those run in FP32 (0.75e-7 off a
// block of three targets, a tile's members 1.1e-7). Returns the pass's cost. search: blocks by first fit or by roll-outs,
// whichever are fewer.
double tc_tile_blocks(int n, const std::vector<qs_gate> &pg, const Pending &pass, int K, bool search, TcPass &out) {
  uint64_t t = pass.tmask | ((1ull << kTileLowBits) - 1);
  for (int q = 0; q < n && popcount64(t) < kTcTileBits; q++) t |= 1ull << q;
  out.tile = t;
  auto fits = [&](uint64_t q) { return popcount64(q & t) <= 5 && popcount64(q & ~t) <= kTcTileSel; };
  const std::vector<int> idx = one_qubit_late(pg, pass.members);
  greedy_groups(pg, idx, out.blocks,
                [&](const Pending &p, int, uint64_t gmask, uint64_t, bool) { return fits(p.qmask | gmask); });
  if (search) {
    std::vector<Pending> alt;
    lookahead_groups(
        pg, idx, alt, [&](const LookGroup &a, const LookGroup &b) { return fits(a.qmask | b.qmask); }, 40, 3,
        true);
    if (alt.size() < out.blocks.size()) out.blocks.swap(alt);
  }
  std::vector<Pending> single;
  greedy_groups(pg, idx, single, [&](const Pending &p, int, uint64_t gmask, uint64_t, bool) {
    return popcount64(p.qmask | gmask) <= K;
  });
  bool fp32 = true;
  for (const Pending &p : single) fp32 = fp32 && popcount64(p.qmask) < 4;
  if (fp32 || (double)single.size() <= tc_tile_cost(out.blocks.size())) {
    out.single = true;
    out.blocks.swap(single);
    return (double)out.blocks.size();
  }
  return tc_tile_cost(out.blocks.size());
}

// The cheapest of a few groupings into passes; returns its cost. The roll-outs
// over blocks save one in seven at 0.4 us of host time a gate, those over
// passes one pass and one block in ten more at 3 us: on layered circuits a
// launch of a single block takes 30, 60, 120 and 250 us at 23 to 26 qubits, so
// that the first pay from 23 qubits on and the second from 26.
constexpr int kPassSearchBits = 26;

double tc_tile_passes(int n, const std::vector<qs_gate> &pg, const std::vector<int> &all, int K, bool search,
                      std::vector<TcPass> &out) {
  const uint64_t low = (1ull << kTileLowBits) - 1;
  auto first_fit = [&](std::vector<Pending> &passes) {
    greedy_groups(pg, all, passes, [&](const Pending &p, int, uint64_t, uint64_t gt, bool) {
      return popcount64(p.tmask | low | gt) <= kTcTileBits;
    });
  };
  if (!search || n < kPassSearchBits) {
    std::vector<Pending> passes;
    first_fit(passes);
    out.resize(passes.size());
    std::vector<double> cost(passes.size());
    parallel_for(passes.size(), search ? 0.4 * (double)all.size() : 0.0,
                 [&](size_t i) { cost[i] = tc_tile_blocks(n, pg, passes[i], K, search, out[i]); });
    double total = 0;
    for (double c : cost) total += c;
    return total;
  }
  struct Variant {
    int horizon, tail;
  };
  const Variant variants[] = {{0, 0}, {60, 1}, {60, 2}, {40, 2}};
  std::vector<TcPass> alt[4];
  double total[4] = {0, 0, 0, 0};
  parallel_for(4, 9.0 * roll_out_gates(all.size(), 60), [&](size_t v) {
    std::vector<Pending> passes;
    if (v == 0) {
      first_fit(passes);
    } else {
      lookahead_groups(
          pg, all, passes,
          [&](const LookGroup &a, const LookGroup &b) { return popcount64(a.tmask | low | b.tmask) <= kTcTileBits; },
          variants[v].horizon, variants[v].tail, false);
    }
    alt[v].resize(passes.size());
    for (size_t i = 0; i < passes.size(); i++) total[v] += tc_tile_blocks(n, pg, passes[i], K, true, alt[v][i]);
  });
  size_t best = 0;
  for (size_t v = 1; v < 4; v++)
    if (total[v] < total[best]) best = v;
  out.swap(alt[best]);
  return total[best];
}

// A member of a tensor-core tile pass; false when all its gates are the
// identity.
bool finish_tile_member(const std::vector<qs_gate> &pg, const Pending &p, uint64_t tile, Block &out) {
  out = Block();
  out.kind = BK_DENSE;
  out.k = 5;
  out.n_gates = (int)p.members.size();
  uint64_t t = p.qmask & tile;
  for (int q = 0; popcount64(t) < 5; q++)  // widened by an identity, bit 0 first (16-byte accesses)
    if ((tile >> q) & 1) t |= 1ull << q;
  int w = 0;
  for (int q = 0; q < 64; q++) {
    if ((t >> q) & 1) out.q[w++] = q;
    if ((p.qmask & ~tile) >> q & 1) out.sel[out.nsel++] = q;
  }
  const int variants = 1 << out.nsel;
  out.skip = (1u << variants) - 1;
  out.gates.reserve(p.members.size());
  std::vector<cd> G;
  for (int gi : p.members) {
    const qs_gate &g = pg[gi];
    gate_full_matrix(g, G);
    const int d = 1 << g.nq;
    Block::Member m = {(int8_t)g.nq, {0, 0, 0}};
    for (int j = 0; j < g.nq; j++) {
      const int at = pos_of(out.q, 5, g.q[j]);
      m.at[j] = (int8_t)(at >= 0 ? at : -1 - pos_of(out.sel, out.nsel, g.q[j]));
    }
    // the variants in which the gate does something: rows and columns with
    // the outer bits at the variant's values
    for (int v = 0; v < variants; v++) {
      if (!((out.skip >> v) & 1)) continue;
      bool identity = true;
      for (int r = 0; r < d && identity; r++) {
        bool in = true;
        for (int j = 0; j < g.nq; j++)
          if (m.at[j] < 0 && ((r >> j) & 1) != ((v >> (-1 - m.at[j])) & 1)) in = false;
        for (int c = 0; c < d && in && identity; c++) {
          const cd z = G[(size_t)r * d + c];
          identity = r == c ? is_one(z) : is_zero(z);
        }
      }
      if (!identity) out.skip &= ~(1u << v);
    }
    out.mat.insert(out.mat.end(), G.begin(), G.end());
    out.gates.push_back(m);
  }
  return out.skip != (1u << variants) - 1;
}

// Fusion and classification of the physical gates pg[idx...] (one segment
// of the circuit between global-tier exchanges); appends the blocks.
qs_status plan_segment(int n, const std::vector<qs_gate> &pg, const std::vector<int> &all, uint64_t flags,
                       const qs_opts &opts, int D, int K, bool c128, bool allow_phase, bool repeated, bool tc_tiles,
                       std::vector<Block> &plan, std::string &err) {
  const bool fuse = flags & QS_FUSE;
  const bool dfuse = flags & QS_DIAG;
  std::vector<Pending> groups;
  std::vector<TcPass> passes;
  bool tiled_tc = false;
  double tiled_cost = 0;
  const bool tiled = (flags & QS_TILE) && n > tile_bits_of(opts, c128);
  if (tiled) {
    std::vector<Block> tplan;
    qs_status ts = tile_plan(n, pg, all, opts, c128, repeated, tplan, err);
    if (ts != QS_OK) return ts;
    for (Block &b : tplan) plan.push_back(std::move(b));
    return QS_OK;
  }
  if (!fuse && !dfuse) {
    groups.resize(all.size());
    for (size_t i = 0; i < all.size(); i++) {
      const qs_gate &g = pg[all[i]];
      groups[i].members.push_back(all[i]);
      for (int j = 0; j < g.nq; j++) groups[i].qmask |= 1ull << g.q[j];
      groups[i].all_diag = op_info(g.op).diagonal;
    }
  } else {
    // diagonal runs: up to D qubits as a phase table, any width as a phase
    // polynomial (states of at least 11 qubits, which the kernel needs)
    const bool phase_ok = dfuse && allow_phase && n > QS_MAX_DIAG;
    const int dlimit = phase_ok ? 64 : D;
    auto limit = [&](bool nd) { return nd ? (dfuse ? dlimit : std::max(K, 1)) : K; };
    auto fits = [&](const LookGroup &a, const LookGroup &b) {
      return popcount64(a.qmask | b.qmask) <= limit(a.all_diag && b.all_diag);
    };
    auto first_fit = [&](std::vector<Pending> &g) {
      greedy_groups(pg, all, g, [&](const Pending &p, int, uint64_t gmask, uint64_t, bool gdiag) {
        return popcount64(p.qmask | gmask) <= limit(p.all_diag && gdiag);
      });
    };
    // The search saves one block in six on layered circuits, so it has to
    // cost less than that share of the passes. Roll-outs with free joins cost
    // about 1 us of host time per gate, and a gate about a twelfth of a pass:
    // they pay from 23 qubits on (20 us a pass in complex64; complex128
    // passes take five times as long and pay from 22 on), or where a plan is
    // run again and again (a batch). Without free joins they cost 5 us per
    // gate and sometimes save a few blocks more at 6 targets (98 instead of
    // 107 for the 30-qubit random circuit): from 27 qubits on (25). A caller
    // that asks for another horizon than the default gets all of it.
    const int wide = n + (c128 ? 1 : 0);
    const bool asked = opts.fuse_lookahead > 0 && opts.fuse_lookahead != kLookahead;
    const bool search = opts.fuse_lookahead > 0 && (wide >= kSearchBits || repeated || asked);
    first_fit(groups);
    // (a circuit of one block gains nothing from a tile: three targets at 26
    // qubits 341 us with the call's host time, 323 us by itself, at 16 qubits
    // 91 and 30 us)
    if (tc_tiles && groups.size() > 1) {
      // Roll-outs cost by the gate and gain by the block: not where a block
      // has many gates (all pairs of 26 qubits in one diagonal run, 325 gates,
      // lost 0.5 ms to them). Layered circuits have 11 to 14 gates to a block.
      const double block_gates = std::ldexp(16.0, n - (n < kPassSearchBits ? kSearchBits : kPassSearchBits));
      const bool roll_outs = asked || (search && (double)all.size() <= block_gates * (double)groups.size());
      tiled_cost = tc_tile_passes(n, pg, all, K, roll_outs, passes);
      // not searched where no search (it saves one block in six) would change the choice
      tiled_tc = tiled_cost < (search ? 0.8 : 1.0) * (double)groups.size();
    }
    if (search && !tiled_tc && groups.size() > 1) {
      // no horizon or tie-break (by the width of the last 6 or 12 blocks) is
      // best on every circuit: first fit and several roll-outs run side by
      // side on host threads, and the grouping with the fewest blocks is
      // launched (the earliest on a tie)
      struct Variant {
        int horizon, tail;
        bool free_joins;
      };
      const int L = opts.fuse_lookahead;
      const Variant variants[] = {{0, 0, false},          {L, 6, true},       {L, 12, true},
                                  {L + L / 3, 6, true},   {L, 6, false},      {L, 12, false},
                                  {L + L / 3, 6, false},  {L + L / 3, 12, false}, {L + 2 * L / 3, 6, false}};
      const size_t count = n + (c128 ? 2 : 0) >= kFullSearchBits || asked ? 9 : 4;
      std::vector<std::vector<Pending>> alt(count);
      auto one = [&](size_t v) {
        if (v == 0) alt[0] = groups;
        else lookahead_groups(pg, all, alt[v], fits, variants[v].horizon, variants[v].tail, variants[v].free_joins);
      };
      // (in batches many circuits are planned one after the other: threads would cost more than they save)
      parallel_for(count, repeated ? 0 : (count > 4 ? 20.0 : 3.0) * roll_out_gates(all.size(), L), one);
      size_t best = 0;
      for (size_t v = 1; v < count; v++)
        if (alt[v].size() < alt[best].size()) best = v;
      groups.swap(alt[best]);
      tiled_tc = tc_tiles && tiled_cost < (double)groups.size();
    }
  }

  // (2b) tensor-core tile passes instead, where they cost less
  if (tiled_tc) {
    std::vector<std::pair<size_t, size_t>> at;  // (pass, block)
    double us = 0;
    for (size_t i = 0; i < passes.size(); i++)
      for (size_t j = 0; j < passes[i].blocks.size(); j++) {
        const Pending &p = passes[i].blocks[j];
        at.push_back({i, j});
        us += (passes[i].single ? 1.3 : 0.3) * (double)p.members.size();
      }
    std::vector<Block> done(at.size());
    std::vector<char> keep(at.size(), 0);
    parallel_for(at.size(), us, [&](size_t x) {
      const TcPass &t = passes[at[x].first];
      const Pending &p = t.blocks[at[x].second];
      keep[x] = t.single ? finish_block(pg, p, true, done[x], D) : finish_tile_member(pg, p, t.tile, done[x]);
    });
    for (size_t x = 0; x < at.size();) {
      const size_t i = at[x].first;
      if (passes[i].single) {
        if (keep[x]) plan.push_back(std::move(done[x]));
        x++;
        continue;
      }
      Block b;
      auto open = [&] {
        b = Block();
        b.kind = BK_TILE;
        b.tc = true;
        b.k = kTcTileBits;
        b.meta = 5;
        int w = 0;
        for (int q = 0; q < 64; q++)
          if ((passes[i].tile >> q) & 1) b.tile_q[w++] = q;
      };
      open();
      for (; x < at.size() && at[x].first == i; x++) {
        if (!keep[x]) continue;
        if (b.sub.size() == (size_t)kTcTileMaxBlocks) {
          plan.push_back(std::move(b));
          open();
        }
        b.n_gates += done[x].n_gates;
        b.sub.push_back(std::move(done[x]));
      }
      if (!b.sub.empty()) plan.push_back(std::move(b));
    }
    return QS_OK;
  }

  // (3) products and classification
  std::vector<Block> done(groups.size());
  std::vector<char> keep(groups.size(), 0);
  const bool phase_ok = dfuse && allow_phase && n > QS_MAX_DIAG;
  parallel_for(groups.size(), repeated ? 0 : products_us(groups), [&](size_t i) {
    if (!groups[i].members.empty()) keep[i] = finish_block(pg, groups[i], true, done[i], D, phase_ok) ? 1 : 0;
  });
  for (size_t i = 0; i < groups.size(); i++)
    if (keep[i]) plan.push_back(std::move(done[i]));
  return QS_OK;
}

int digit_check(const std::vector<cd> &m) {
  const double least = std::ldexp(1.0, -2 * kDigitSpan);
  int check = 0;
  for (const cd &z : m) {
    const double s = std::norm(z);
    if (s < least) check = std::max(check, z == cd(0, 0) ? 1 : 2);
  }
  return check;
}

}  // namespace

void parallel_blocks(size_t n, double work_us, const std::function<void(size_t)> &f) { parallel_for(n, work_us, f); }

int tile_bits_of(const qs_opts &o, bool c128) {
  if (o.tile_bits > 0) return std::min(o.tile_bits, c128 ? kMaxTileBits - 1 : kMaxTileBits);
  return c128 ? 12 : 13;  // 64 KiB of amplitudes
}

int tile_k_of(const qs_opts &o) { return o.tile_k > 0 ? std::min(o.tile_k, 4) : 3; }

void fill_record(const Block &b, int index, int n, int amp_bytes, qs_block_record &r) {
  std::memset(&r, 0, sizeof(r));
  r.index = (int32_t)index;
  r.kind = (uint8_t)b.kind;
  r.k = (uint8_t)b.k;
  r.nctrl = (uint8_t)b.nctrl;
  r.tc = b.tc ? (b.tc_xg ? 2 : 1) : 0;
  for (int j = 0; j < QS_MAX_DIAG; j++) r.qubits[j] = j < b.k ? (int8_t)b.q[j] : (int8_t)-1;
  if (b.kind == BK_TILE)
    for (int j = 0; j < QS_MAX_DIAG; j++)
      r.qubits[j] = kTileLowBits + j < b.k ? (int8_t)b.tile_q[kTileLowBits + j] : (int8_t)-1;
  r.meta = (uint8_t)b.meta;
  r.op = b.n_gates == 1 ? (uint8_t)b.first_op : (uint8_t)255;
  r.n_gates = b.n_gates;
  r.cmask = b.cmask;
  r.bytes = block_bytes(b, n, amp_bytes);
  r.t_start_ms = -1;
  r.ms = -1;
}

bool tc_tiles_apply(int n, bool c128, uint64_t flags, uint64_t chosen, const qs_opts &o) {
  return (flags & QS_PGO_RULES) && !(flags & (QS_PGO_MEASURED | QS_PROFILE)) && (chosen & QS_TC) && !c128 &&
         n > kTcTileBits && o.threads == 0 && o.tc_exchange == 0 && o.tc_precision == 0 && o.n_global == 0;
}

Block tile_member_block(const Block &m) {
  // the qubits that some gate acts on, ascending: its targets without the
  // identity's, and the bits outside the tile
  auto qubit = [&](int at) { return at >= 0 ? m.q[at] : m.sel[-1 - at]; };
  uint64_t mask = 0;
  for (const Block::Member &g : m.gates)
    for (int j = 0; j < g.nq; j++) mask |= 1ull << qubit(g.at[j]);
  Block out;
  out.kind = BK_DENSE;
  out.tc = true;
  out.n_gates = m.n_gates;
  for (int q = 0; q < 64; q++)
    if ((mask >> q) & 1) out.q[out.k++] = q;
  Product M(out.k);
  size_t at = 0;
  for (const Block::Member &g : m.gates) {
    const size_t entries = (size_t)1 << (2 * g.nq);
    const std::vector<cd> G(m.mat.begin() + (long)at, m.mat.begin() + (long)(at + entries));
    int pos[3] = {0, 0, 0};
    for (int j = 0; j < g.nq; j++) pos[j] = pos_of(out.q, out.k, qubit(g.at[j]));
    left_multiply(M, G, pos, g.nq);
    at += entries;
  }
  const int d = 1 << out.k;
  out.mat.resize((size_t)d * d);
  for (int r = 0; r < d; r++)
    for (int c = 0; c < d; c++) out.mat[(size_t)r * d + c] = M.at(r, c);
  return out;
}

double block_bytes(const Block &b, int n, int amp_bytes) {
  double amps = std::ldexp(1.0, n - b.nctrl);
  if (b.kind == BK_PERMUTE || b.kind == BK_GLOBAL) amps = std::ldexp(1.0, n - 1);
  return 2.0 * amps * amp_bytes;
}

qs_status build_plan(int n, const qs_gate *gates, size_t n_gates, uint64_t flags,
                     const qs_opts &opts, int8_t *perm, std::vector<Block> &plan,
                     PlanStats &stats, std::string &err, bool c128, bool allow_phase, bool repeated, bool tc_tiles) {
  plan.clear();
  stats = PlanStats();
  stats.gates_in = (int)n_gates;
  // validation first: a bad gate leaves perm untouched
  for (size_t i = 0; i < n_gates; i++) {
    const qs_gate &g = gates[i];
    if (g.op >= QS_N_GATE_TYPES) {
      err = "gate " + std::to_string(i) + ": unknown op";
      return QS_EINVAL;
    }
    if (g.nq != op_info(g.op).nq) {
      err = "gate " + std::to_string(i) + ": qubit count does not match the op";
      return QS_EINVAL;
    }
    for (int j = 0; j < g.nq; j++) {
      if (g.q[j] >= n) {
        err = "gate " + std::to_string(i) + ": qubit out of range";
        return QS_EINVAL;
      }
      for (int k = 0; k < j; k++)
        if (g.q[k] == g.q[j]) {
          err = "gate " + std::to_string(i) + ": duplicate qubit";
          return QS_EINVAL;
        }
    }
    for (int j = 0; j < op_info(g.op).nparams; j++)
      if (!std::isfinite(g.p[j])) {
        err = "gate " + std::to_string(i) + ": non-finite angle";
        return QS_EINVAL;
      }
  }
  const bool vswap = flags & QS_VSWAP;
  const bool fuse = flags & QS_FUSE;
  int K = fuse ? QS_FUSE_K_OF(flags) : 0;
  if (fuse && K == 0) K = 4;
  if (K > QS_MAX_FUSE) {
    err = "fusion width above QS_MAX_FUSE";
    return QS_EUNSUPPORTED;
  }
  int D = std::max(1, std::min(opts.diag_max, QS_MAX_DIAG));
  if (opts.tc_exchange < 0 || opts.tc_exchange > 2) {
    err = "opts.tc_exchange out of range (0..2)";
    return QS_EINVAL;
  }
  if (opts.tc_max_ctas < 0) {
    err = "opts.tc_max_ctas must not be negative";
    return QS_EINVAL;
  }
  if (opts.n_global < 0 || opts.n_global > n - 1 || (opts.n_global > 0 && n - opts.n_global < 2)) {
    err = "opts.n_global out of range (0..n-2 global bits, two local bits at least)";
    return QS_EINVAL;
  }
  if (flags & QS_TILE) {
    const int tmax = c128 ? kMaxTileBits - 1 : kMaxTileBits;
    if (opts.tile_bits != 0 && (opts.tile_bits < 8 || opts.tile_bits > tmax)) {
      err = "opts.tile_bits out of range";
      return QS_EINVAL;
    }
    if (opts.tile_k < 0 || opts.tile_k > 4) {
      err = "opts.tile_k out of range (0..4)";
      return QS_EINVAL;
    }
  }

  // (0) rotation folding (an IR rewrite; exact)
  std::vector<qs_gate> folded;
  if (flags & QS_FOLD) {
    folded = fold_rotations(n, gates, n_gates);
    stats.gates_removed = (int)n_gates - (int)folded.size();
    gates = folded.data();
    n_gates = folded.size();
  }

  // (1) virtual swap and renaming to physical qubits
  std::vector<qs_gate> pg;
  pg.reserve(n_gates);
  for (size_t i = 0; i < n_gates; i++) {
    qs_gate g = gates[i];
    if (vswap && g.op == QS_SWAP) {
      std::swap(perm[g.q[0]], perm[g.q[1]]);
      stats.swaps_absorbed++;
      continue;
    }
    for (int j = 0; j < g.nq; j++) g.q[j] = (uint8_t)perm[g.q[j]];
    pg.push_back(g);
  }

  // (1b) relocation (Sec. III-D: move hot qubits out of the slow segment).
  // Here the slow positions are physical bits 0 and 1: a block whose targets
  // include both gathers 8-byte elements at 32-byte strides. When the share
  // of multi-qubit non-diagonal gates touching them exceeds reloc_share and
  // twice the share a random qubit pair would have, each
  // hot low bit is exchanged once, up front, with the high bit that carries
  // the fewest such gates, and every gate is renamed.
  std::vector<std::pair<int, int>> reloc;
  if ((flags & QS_RELOCATE) && n >= 6) {
    std::vector<double> heat(64, 0.0);
    double total = 0, low = 0;
    for (const qs_gate &g : pg) {
      if (op_info(g.op).diagonal || g.nq < 2) continue;
      total += 1;
      bool touches_low = false;
      for (int j = 0; j < g.nq; j++) {
        heat[g.q[j]] += 1;
        touches_low |= g.q[j] < 2;
      }
      if (touches_low) low += 1;
    }
    // "hot" means well above the share a random pair of qubits would have
    const double uniform = 1.0 - (double)(n - 2) * (n - 3) / ((double)n * (n - 1));
    if (total > 0 && low / total > std::max(opts.reloc_share, 2.0 * uniform)) {
      std::vector<int> used;
      for (int lowq = 0; lowq < 2; lowq++) {
        if (heat[lowq] == 0) continue;
        int best = -1;
        for (int q = n - 1 - opts.n_global; q >= 5; q--) {
          if (std::find(used.begin(), used.end(), q) != used.end()) continue;
          if (best < 0 || heat[q] < heat[best]) best = q;
        }
        if (best < 0 || heat[best] >= heat[lowq]) continue;
        used.push_back(best);
        reloc.push_back({lowq, best});
      }
      for (auto &pr : reloc) {
        const int a = pr.first, b = pr.second;
        for (qs_gate &g : pg)
          for (int j = 0; j < g.nq; j++) {
            if (g.q[j] == a) g.q[j] = (uint8_t)b;
            else if (g.q[j] == b) g.q[j] = (uint8_t)a;
          }
        for (int l = 0; l < n; l++) {
          if (perm[l] == a) perm[l] = (int8_t)b;
          else if (perm[l] == b) perm[l] = (int8_t)a;
        }
      }
      stats.relocations = (int)reloc.size();
    }
  }

  // (1c) global tier: the top n_global physical bits are held by other
  // ranks (one shard per value of those bits). A gate acting non-diagonally
  // on a global bit first needs that bit exchanged with a local one (a
  // virtual swap of the two bits: a pairwise half-shard exchange between the
  // ranks that differ in the global bit); the plan records the exchange and
  // every later gate, and perm, follow the relabelling. The local bit taken
  // is the one whose next non-diagonal use lies furthest ahead (never used
  // again first; ties: the highest bit), so that exchanges stay rare. Gates
  // that are diagonal on a global bit (controls, phases) need no exchange: a
  // shard knows its global bits.
  std::vector<size_t> cuts;                   // segment starts in pg
  std::vector<std::pair<int, int>> gswaps;    // (local, global) exchanged at each cut
  const int nloc = n - opts.n_global;
  if (opts.n_global > 0) {
    auto next_use = [&](size_t from, int q) {
      for (size_t i = from; i < pg.size(); i++)
        for (int j = 0; j < pg[i].nq; j++)
          if (pg[i].q[j] == q && !gate_diag_on(pg[i], j)) return i;
      return pg.size();
    };
    for (size_t i = 0; i < pg.size(); i++) {
      for (int j = 0; j < pg[i].nq; j++) {
        const int G = pg[i].q[j];
        if (G < nloc || gate_diag_on(pg[i], j)) continue;
        int L = -1;
        size_t far = 0;
        for (int q = nloc - 1; q >= 0; q--) {
          bool in_gate = false;
          for (int jj = 0; jj < pg[i].nq; jj++) in_gate |= pg[i].q[jj] == q;
          if (in_gate) continue;
          const size_t u = next_use(i, q);
          if (L < 0 || u > far) {
            L = q;
            far = u;
          }
        }
        if (L < 0) {
          err = "global tier: no local bit free for an exchange";
          return QS_EUNSUPPORTED;
        }
        for (size_t k2 = i; k2 < pg.size(); k2++)
          for (int jj = 0; jj < pg[k2].nq; jj++) {
            if (pg[k2].q[jj] == G) pg[k2].q[jj] = (uint8_t)L;
            else if (pg[k2].q[jj] == L) pg[k2].q[jj] = (uint8_t)G;
          }
        for (int l = 0; l < n; l++) {
          if (perm[l] == G) perm[l] = (int8_t)L;
          else if (perm[l] == L) perm[l] = (int8_t)G;
        }
        cuts.push_back(i);
        gswaps.push_back({L, G});
      }
    }
  }

  push_exchanges(reloc, plan);
  size_t seg_begin = 0;
  for (size_t sgi = 0; sgi <= cuts.size(); sgi++) {
    const size_t seg_end = sgi < cuts.size() ? cuts[sgi] : pg.size();
    std::vector<int> idx;
    for (size_t i = seg_begin; i < seg_end; i++) idx.push_back((int)i);
    qs_status st = plan_segment(n, pg, idx, flags, opts, D, K, c128, allow_phase, repeated, tc_tiles, plan, err);
    if (st != QS_OK) return st;
    if (sgi < cuts.size()) {
      Block b;
      b.kind = BK_GLOBAL;
      b.k = 2;
      b.q[0] = gswaps[sgi].first;
      b.q[1] = gswaps[sgi].second;
      b.n_gates = 0;
      b.meta = 3;
      plan.push_back(std::move(b));
    }
    seg_begin = seg_end;
  }
  const bool tf32 = opts.tc_precision == 1;
  for (Block &b : plan) {
    if (b.kind == BK_TILE && b.tc) {
      b.withhold_commit = opts.test_wait_timeout != 0;
      b.tc_max_ctas = opts.tc_max_ctas;
      continue;
    }
    // complex128 blocks run on FP16 digit planes (tc64.cu), 4 and 5 targets,
    // or keep the FP64 kernel where the options ask for the other precision
    b.tc = (flags & QS_TC) && b.kind == BK_DENSE && b.k >= 4 && b.k <= (tf32 || c128 ? 5 : 6) && !(c128 && tf32);
    if (b.tc && c128) b.digit_check = digit_check(b.mat);
    b.tc_tf32 = b.tc && tf32;
    b.shuffles = opts.no_shuffles == 0;
    // lane-exchange gathers where they measured faster (tc_exchange_pays),
    // or everywhere the layout allows with tc_exchange = 2
    TcXLayout xl;
    b.tc_xg = b.tc && !tf32 && !c128 && opts.tc_exchange != 1 && (opts.tc_exchange == 2 || tc_exchange_pays(b)) &&
              tc_exchange_layout(n, b, xl);
    b.withhold_commit = b.tc && opts.test_wait_timeout != 0;
    b.tc_max_ctas = (b.tc || b.kind == BK_PHASE) ? opts.tc_max_ctas : 0;
  }
  return QS_OK;
}

}  // namespace qs
