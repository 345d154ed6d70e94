// Host setup, part 1: fill-reducing ordering and supernodal symbolic analysis
// of the SPD matrices that Alg. 2 factors once, X1 = C + gamma G and G: for
// R-MATEX X1 = C + gamma G (Sec. 3.3.2), and G itself for F, P and the DC
// state (Eq. 6).  C is diagonal, so both share one sparsity pattern and one
// symbolic analysis.
//
// Ordering: recursive nested dissection with breadth-first level-structure
// separators (no coordinates are needed, only the graph of G).
#include <algorithm>
#include <cstring>
#include <numeric>

#include "internal.h"

namespace matex {

namespace {

struct Graph {
  int64_t n;
  std::vector<int64_t> ptr;
  std::vector<int32_t> adj;
};

Graph build_graph(const CsrSym& A) {
  Graph g;
  g.n = A.n;
  g.ptr.assign(A.n + 1, 0);
  for (int64_t i = 0; i < A.n; ++i) {
    int64_t cnt = 0;
    for (int64_t p = A.rowptr[i]; p < A.rowptr[i + 1]; ++p)
      if (A.col[p] != i) ++cnt;
    g.ptr[i + 1] = g.ptr[i] + cnt;
  }
  g.adj.resize(g.ptr[A.n]);
  for (int64_t i = 0; i < A.n; ++i) {
    int64_t q = g.ptr[i];
    for (int64_t p = A.rowptr[i]; p < A.rowptr[i + 1]; ++p)
      if (A.col[p] != i) g.adj[q++] = A.col[p];
  }
  return g;
}

struct NdState {
  const Graph* g;
  std::vector<int32_t> tag;     // subset membership tag per node
  std::vector<int32_t> level;   // BFS level per node
  std::vector<int32_t> queue;
  int32_t next_tag = 1;
  std::vector<int32_t>* out;
};

// BFS from root over nodes carrying tag t; fills st.queue with the visit order
// and st.level; returns the number of levels.
int32_t bfs(NdState& st, int32_t root, int32_t t) {
  const Graph& g = *st.g;
  st.queue.clear();
  st.queue.push_back(root);
  st.level[root] = 0;
  int32_t lvl_tag = -t;  // visited nodes carry -t while the BFS runs
  st.tag[root] = lvl_tag;
  size_t head = 0;
  int32_t maxl = 0;
  while (head < st.queue.size()) {
    int32_t v = st.queue[head++];
    int32_t lv = st.level[v];
    for (int64_t p = g.ptr[v]; p < g.ptr[v + 1]; ++p) {
      int32_t u = g.adj[p];
      if (st.tag[u] == t) {
        st.tag[u] = lvl_tag;
        st.level[u] = lv + 1;
        maxl = std::max(maxl, lv + 1);
        st.queue.push_back(u);
      }
    }
  }
  for (int32_t v : st.queue) st.tag[v] = t;  // restore membership
  return maxl + 1;
}

const int32_t kLeaf = 48;

void nd_rec(NdState& st, std::vector<int32_t>& nodes) {
  if ((int64_t)nodes.size() <= kLeaf) {
    st.out->insert(st.out->end(), nodes.begin(), nodes.end());
    return;
  }
  const Graph& g = *st.g;
  int32_t t = st.next_tag++;
  for (int32_t v : nodes) st.tag[v] = t;
  // pseudo-peripheral root: repeat BFS from the last-visited node
  int32_t root = nodes[0];
  int32_t nl = bfs(st, root, t);
  if (st.queue.size() < nodes.size()) {
    // disconnected subset: order the reached component, then the rest
    std::vector<int32_t> comp(st.queue.begin(), st.queue.end());
    int32_t ct = st.next_tag++;
    for (int32_t v : comp) st.tag[v] = ct;
    std::vector<int32_t> rest;
    rest.reserve(nodes.size() - comp.size());
    for (int32_t v : nodes)
      if (st.tag[v] == t) rest.push_back(v);
    nodes.clear();
    nodes.shrink_to_fit();
    nd_rec(st, comp);
    nd_rec(st, rest);
    return;
  }
  for (int it = 0; it < 4; ++it) {
    int32_t cand = st.queue.back();
    int32_t nl2 = bfs(st, cand, t);
    if (nl2 <= nl && it > 0) {
      if (nl2 < nl) bfs(st, root, t);
      break;
    }
    root = cand;
    nl = nl2;
  }
  if (nl < 3) {  // no proper separator (clique-like); keep as a leaf block
    st.out->insert(st.out->end(), nodes.begin(), nodes.end());
    return;
  }
  std::vector<int64_t> cnt(nl, 0);
  for (int32_t v : st.queue) cnt[st.level[v]]++;
  int64_t half = (int64_t)nodes.size() / 2, acc = 0;
  int32_t mid = 1;
  for (int32_t l = 0; l < nl; ++l) {
    if (acc + cnt[l] > half) { mid = l; break; }
    acc += cnt[l];
  }
  mid = std::max(1, std::min(mid, nl - 2));
  std::vector<int32_t> A, B, S;
  for (int32_t v : st.queue) {
    int32_t lv = st.level[v];
    if (lv < mid) A.push_back(v);
    else if (lv > mid) B.push_back(v);
    else {
      // a separator node with no neighbour beyond the separator joins A
      bool touches_b = false;
      for (int64_t p = g.ptr[v]; p < g.ptr[v + 1]; ++p) {
        int32_t u = g.adj[p];
        if (st.tag[u] == t && st.level[u] == mid + 1) { touches_b = true; break; }
      }
      if (touches_b) S.push_back(v); else A.push_back(v);
    }
  }
  nodes.clear();
  nodes.shrink_to_fit();
  nd_rec(st, A);
  nd_rec(st, B);
  st.out->insert(st.out->end(), S.begin(), S.end());
}

// The supernodes that amalgamation left (gone: merged into another), renumbered.
void keep_supernodes(Symbolic& S, std::vector<std::vector<int32_t>>& offrows,
                     std::vector<int32_t>& col2sup, std::vector<int64_t>& zeros,
                     const std::vector<int32_t>& first, const std::vector<char>& gone) {
  std::vector<int32_t> keep;
  for (int32_t t = 0; t < (int32_t)gone.size(); ++t)
    if (!gone[t]) keep.push_back(t);
  std::sort(keep.begin(), keep.end(), [&](int32_t a, int32_t b) { return first[a] < first[b]; });
  std::vector<std::vector<int32_t>> rows2(keep.size());
  std::vector<int64_t> zeros2(keep.size());
  S.sup_first.assign(keep.size() + 1, 0);
  for (size_t k = 0; k < keep.size(); ++k) {
    S.sup_first[k] = first[keep[k]];
    rows2[k].swap(offrows[keep[k]]);
    zeros2[k] = zeros[keep[k]];
  }
  zeros.swap(zeros2);
  S.nsup = (int32_t)keep.size();
  S.sup_first[S.nsup] = (int32_t)S.n;
  for (int32_t t = 0; t < S.nsup; ++t)
    for (int32_t j = S.sup_first[t]; j < S.sup_first[t + 1]; ++j) col2sup[j] = t;
  S.sup_parent.assign(S.nsup, -1);
  for (int32_t t = 0; t < S.nsup; ++t)
    if (!rows2[t].empty()) S.sup_parent[t] = col2sup[rows2[t][0]];
  offrows.swap(rows2);
}

// Supernodes renumbered: every parent's children with the largest subtree
// first, so that the small ones end up adjacent to their parent, and those of
// level l0 and above (lev) after all others.  Only the numbering changes, no
// panel.
void order_children(Symbolic& S, std::vector<std::vector<int32_t>>& offrows,
                    std::vector<int32_t>& col2sup, std::vector<int64_t>& zeros,
                    std::vector<int32_t>& lev, int32_t l0) {
  const int32_t ns = S.nsup;
  std::vector<int64_t> size(ns);
  std::vector<std::vector<int32_t>> kids(ns);
  std::vector<int32_t> stack, order;
  for (int32_t s = 0; s < ns; ++s) size[s] += S.sup_first[s + 1] - S.sup_first[s];
  for (int32_t s = 0; s < ns; ++s)
    if (S.sup_parent[s] >= 0) {  // children come before their parent
      size[S.sup_parent[s]] += size[s];
      kids[S.sup_parent[s]].push_back(s);
    }
  for (int32_t r = ns - 1; r >= 0; --r)
    if (S.sup_parent[r] < 0) stack.push_back(r);
  // parents before children, the largest subtree last; then backwards
  while (!stack.empty()) {
    const int32_t s = stack.back();
    stack.pop_back();
    order.push_back(s);
    std::stable_sort(kids[s].begin(), kids[s].end(),
                     [&](int32_t a, int32_t b) { return size[a] > size[b]; });
    stack.insert(stack.end(), kids[s].begin(), kids[s].end());
  }
  std::reverse(order.begin(), order.end());
  std::stable_partition(order.begin(), order.end(), [&](int32_t s) { return lev[s] < l0; });
  std::vector<int32_t> first(ns + 1, 0), map(S.n), pos(ns), perm(S.n), par(ns), lv(ns);
  std::vector<std::vector<int32_t>> rows(ns);
  std::vector<int64_t> z(ns);
  for (int32_t k = 0; k < ns; ++k) {
    const int32_t s = order[k], w = S.sup_first[s + 1] - S.sup_first[s];
    pos[s] = k;
    first[k + 1] = first[k] + w;
    z[k] = zeros[s];
    lv[k] = lev[s];
    for (int32_t j = 0; j < w; ++j) {
      map[S.sup_first[s] + j] = first[k] + j;
      perm[first[k] + j] = S.perm[S.sup_first[s] + j];
      col2sup[first[k] + j] = k;
    }
  }
  for (int32_t s = 0; s < ns; ++s) {
    par[pos[s]] = S.sup_parent[s] < 0 ? -1 : pos[S.sup_parent[s]];
    std::vector<int32_t>& r = rows[pos[s]];
    r.swap(offrows[s]);
    for (int32_t& i : r) i = map[i];
    std::sort(r.begin(), r.end());
  }
  S.sup_first.swap(first);
  S.sup_parent.swap(par);
  S.perm.swap(perm);
  for (int64_t k = 0; k < S.n; ++k) S.iperm[S.perm[k]] = (int32_t)k;
  offrows.swap(rows);
  zeros.swap(z);
  lev.swap(lv);
}

// Widest merged top: every level taken away saves two dependent launches
// (level solves: 4.5 to 8 us each).  Pair of 8 columns, 512 against none: 77
// against 99 us on 10,000 nodes, 141 against 164 us on 39,711 (1,024: 70 and
// 134).  The limit was set by the solution's error on the latter, 2.2e-15 with
// none, 2.6e-15 with 512, 3.0e-15 with 1,024, which was the factors' (their pivots
// cancelled); on the factors as host_numeric.cpp makes them now it is the same
// with none and with 512 (2.6e-16 in extended-precision products).
constexpr int64_t kTopWidth = 512;
constexpr int64_t kTopMinN = 8192;  // smaller grids keep their panels for the resident rounds

// Level of every supernode: 0 for leaves, else one above its highest child.
std::vector<int32_t> sup_levels(const Symbolic& S) {
  std::vector<int32_t> lev(S.nsup, 0);
  for (int32_t s = 0; s < S.nsup; ++s)
    if (S.sup_parent[s] >= 0) lev[S.sup_parent[s]] = std::max(lev[S.sup_parent[s]], lev[s] + 1);
  return lev;
}

// The lowest level from which the tree above is at most `cap` columns and has
// one root: those supernodes may become one (number of levels: none).
int32_t top_level(const Symbolic& S, const std::vector<int32_t>& lev, int64_t cap) {
  int32_t nlev = 0, roots = 0;
  for (int32_t s = 0; s < S.nsup; ++s) {
    nlev = std::max(nlev, lev[s] + 1);
    roots += S.sup_parent[s] < 0;
  }
  if (roots != 1) return nlev;
  std::vector<int64_t> w(nlev, 0);
  for (int32_t s = 0; s < S.nsup; ++s) w[lev[s]] += S.sup_first[s + 1] - S.sup_first[s];
  int32_t l = nlev;
  for (int64_t sum = 0; l > 0 && sum + w[l - 1] <= cap; --l) sum += w[l - 1];
  return l;
}

// The supernodes of level l0 and above, numbered last, as one.
void merge_top(Symbolic& S, std::vector<std::vector<int32_t>>& offrows, std::vector<int32_t>& col2sup,
               std::vector<int64_t>& zeros, const std::vector<int32_t>& lev, int32_t l0) {
  std::vector<char> gone(S.nsup, 0);
  std::vector<int32_t> first(S.sup_first.begin(), S.sup_first.end() - 1);
  int32_t root = -1;
  int64_t w = 0, have = 0;
  for (int32_t s = 0; s < S.nsup; ++s) {
    if (lev[s] < l0) continue;
    const int64_t ws = S.sup_first[s + 1] - S.sup_first[s];
    if (root < 0) first[S.nsup - 1] = S.sup_first[s];
    root = s;
    w += ws;
    have += ws * (ws + 1) / 2 + ws * (int64_t)offrows[s].size() - zeros[s];
    gone[s] = s != S.nsup - 1;
  }
  if (root < 0) return;
  zeros[root] = w * (w + 1) / 2 - have;
  keep_supernodes(S, offrows, col2sup, zeros, first, gone);
}

// Amalgamation for the tensor-core solves (k_sptrsv_mma.cu), whose unit of
// work is a 16 x 16 block of the panel, on top of the relaxed one: a child
// adjacent to its parent joins it when the merged panel costs no more than the
// two: blocks, plus kRow per panel row (splitting or conversion and atomics of
// its right-hand sides), plus kSup per supernode (a thread block's chain of
// loads).  On the 180k-node grid 4,350 supernodes in 15 levels come from 27,600
// in 18, the blocks grow by a tenth, the panel rows shrink from 683k to 425k;
// kSup of 0.5 to 8 and kRow of 0.05 to 0.2 measured within 5 %, a limit of 0.6
// on the zeros 12 % slower than 0.8.
void amalgamate_tiled(Symbolic& S, std::vector<std::vector<int32_t>>& offrows,
                      std::vector<int32_t>& col2sup, std::vector<int64_t>& zeros, int32_t max_width) {
  constexpr double kRow = 0.12, kSup = 2.0, kMaxZeros = 0.8;
  const int32_t ns = S.nsup;
  std::vector<int32_t> first(S.sup_first.begin(), S.sup_first.end() - 1);
  std::vector<int32_t> last(S.sup_first.begin() + 1, S.sup_first.end());
  std::vector<char> gone(ns, 0);
  std::vector<std::vector<int32_t>> kids(ns);
  for (int32_t t = 0; t < ns; ++t)
    if (S.sup_parent[t] >= 0) kids[S.sup_parent[t]].push_back(t);
  auto cost = [&](int64_t w, int64_t ld) {
    return (double)((w + 15) / 16) * (double)((ld + 15) / 16) + kRow * (double)ld + kSup;
  };
  for (int32_t p = 0; p < ns; ++p) {
    std::vector<int32_t>& ch = kids[p];
    const int64_t rp = (int64_t)offrows[p].size();
    while (!ch.empty()) {
      const int32_t t = ch.back();  // the child that ends where p begins
      if (last[t] != first[p]) break;
      const int64_t ws = last[t] - first[t], wp = last[p] - first[p], w = ws + wp;
      const int64_t rt = (int64_t)offrows[t].size();
      const int64_t z = zeros[t] + zeros[p] + ws * (wp + rp - rt);
      const double dense = (double)w * (double)(w + 1) / 2.0 + (double)w * (double)rp;
      if (w > max_width || (double)z > kMaxZeros * dense ||
          cost(w, w + rp) > cost(ws, ws + rt) + cost(wp, wp + rp))
        break;
      first[p] = first[t];
      zeros[p] = z;
      gone[t] = 1;
      ch.pop_back();
      // its own children are p's now; the last of them may end where p begins
      ch.insert(ch.end(), kids[t].begin(), kids[t].end());
    }
  }
  keep_supernodes(S, offrows, col2sup, zeros, first, gone);
}

// Row lists, panel offsets and levels of the supernodes found.
void lay_out(Symbolic& S, const std::vector<std::vector<int32_t>>& offrows) {
  S.sup_rowptr.assign(S.nsup + 1, 0);
  S.pan_off.assign(S.nsup + 1, 0);
  S.nnz_L = 0;
  S.flops_factor = 0;
  for (int32_t s = 0; s < S.nsup; ++s) {
    int64_t w = S.sup_first[s + 1] - S.sup_first[s];
    int64_t r = (int64_t)offrows[s].size();
    S.sup_rowptr[s + 1] = S.sup_rowptr[s] + w + r;
    S.pan_off[s + 1] = S.pan_off[s] + (w + r) * w;
    S.nnz_L += w * (w - 1) / 2 + w * r;
    double nr = (double)(w + r);
    S.flops_factor += (double)w * nr * nr;  // order of the partial factorisation cost
  }
  S.sup_rows.resize(S.sup_rowptr[S.nsup]);
  for (int32_t s = 0; s < S.nsup; ++s) {
    int64_t q = S.sup_rowptr[s];
    for (int32_t j = S.sup_first[s]; j < S.sup_first[s + 1]; ++j) S.sup_rows[q++] = j;
    for (int32_t i : offrows[s]) S.sup_rows[q++] = i;
  }
  // levels of the supernodal tree, leaves first
  std::vector<int32_t> lev(S.nsup, 0);
  int32_t maxlev = 0;
  for (int32_t s = 0; s < S.nsup; ++s) {
    int32_t p = S.sup_parent[s];
    if (p >= 0) lev[p] = std::max(lev[p], lev[s] + 1);
    maxlev = std::max(maxlev, lev[s]);
  }
  S.level_ptr.assign(maxlev + 2, 0);
  for (int32_t s = 0; s < S.nsup; ++s) S.level_ptr[lev[s] + 1]++;
  for (int32_t l = 0; l <= maxlev; ++l) S.level_ptr[l + 1] += S.level_ptr[l];
  S.level_sups.resize(S.nsup);
  {
    std::vector<int32_t> fill(S.level_ptr.begin(), S.level_ptr.end() - 1);
    for (int32_t s = 0; s < S.nsup; ++s) S.level_sups[fill[lev[s]]++] = s;
  }
}

}  // namespace

std::string nested_dissection(const CsrSym& A, std::vector<int32_t>& perm) {
  Graph g = build_graph(A);
  NdState st;
  st.g = &g;
  st.tag.assign(A.n, 0);
  st.level.assign(A.n, 0);
  std::vector<int32_t> out;
  out.reserve(A.n);
  st.out = &out;
  std::vector<int32_t> all(A.n);
  std::iota(all.begin(), all.end(), 0);
  nd_rec(st, all);
  if ((int64_t)out.size() != A.n) return "nested dissection lost nodes";
  perm.swap(out);
  return "";
}

std::string symbolic_analysis(const CsrSym& A, const std::vector<int32_t>& nd_perm,
                              int32_t max_width, Symbolic& S, Symbolic* coarse) {
  const int64_t n = A.n;
  std::vector<int32_t> ip(n);
  for (int64_t k = 0; k < n; ++k) ip[nd_perm[k]] = (int32_t)k;
  // lower pattern by rows (new numbering): row j lists k < j with A[j,k] != 0
  auto row_lower = [&](const std::vector<int32_t>& perm, const std::vector<int32_t>& iperm,
                       std::vector<int64_t>& rp, std::vector<int32_t>& ci) {
    rp.assign(n + 1, 0);
    for (int64_t j = 0; j < n; ++j) {
      int32_t o = perm[j];
      int64_t c = 0;
      for (int64_t p = A.rowptr[o]; p < A.rowptr[o + 1]; ++p)
        if (iperm[A.col[p]] < j) ++c;
      rp[j + 1] = rp[j] + c;
    }
    ci.resize(rp[n]);
    for (int64_t j = 0; j < n; ++j) {
      int32_t o = perm[j];
      int64_t q = rp[j];
      for (int64_t p = A.rowptr[o]; p < A.rowptr[o + 1]; ++p) {
        int32_t k = iperm[A.col[p]];
        if (k < j) ci[q++] = k;
      }
    }
  };
  std::vector<int64_t> rp;
  std::vector<int32_t> ci;
  row_lower(nd_perm, ip, rp, ci);
  // elimination tree (Liu, with path compression)
  std::vector<int32_t> parent(n, -1), anc(n, -1);
  for (int64_t j = 0; j < n; ++j) {
    for (int64_t p = rp[j]; p < rp[j + 1]; ++p) {
      int32_t i = ci[p];
      while (i != -1 && i < j) {
        int32_t nx = anc[i];
        anc[i] = (int32_t)j;
        if (nx == -1) { parent[i] = (int32_t)j; break; }
        i = nx;
      }
    }
  }
  // postorder of the etree (children visited in increasing order)
  std::vector<int32_t> head(n, -1), nxt(n, -1), post;
  post.reserve(n);
  for (int64_t j = n - 1; j >= 0; --j)
    if (parent[j] != -1) { nxt[j] = head[parent[j]]; head[parent[j]] = (int32_t)j; }
  std::vector<int32_t> stk;
  for (int64_t r = 0; r < n; ++r) {
    if (parent[r] != -1) continue;
    stk.push_back((int32_t)r);
    while (!stk.empty()) {
      int32_t v = stk.back();
      if (head[v] != -1) {
        int32_t c = head[v];
        head[v] = nxt[c];
        stk.push_back(c);
      } else {
        post.push_back(v);
        stk.pop_back();
      }
    }
  }
  if ((int64_t)post.size() != n) return "etree postorder failed";
  S.n = n;
  S.perm.resize(n);
  S.iperm.resize(n);
  for (int64_t k = 0; k < n; ++k) S.perm[k] = nd_perm[post[k]];
  for (int64_t k = 0; k < n; ++k) S.iperm[S.perm[k]] = (int32_t)k;
  // everything again in the final numbering
  row_lower(S.perm, S.iperm, rp, ci);
  std::fill(parent.begin(), parent.end(), -1);
  std::fill(anc.begin(), anc.end(), -1);
  for (int64_t j = 0; j < n; ++j) {
    for (int64_t p = rp[j]; p < rp[j + 1]; ++p) {
      int32_t i = ci[p];
      while (i != -1 && i < j) {
        int32_t nx = anc[i];
        anc[i] = (int32_t)j;
        if (nx == -1) { parent[i] = (int32_t)j; break; }
        i = nx;
      }
    }
  }
  // column counts through row subtrees
  std::vector<int64_t> cc(n, 1);
  std::vector<int32_t> mark(n, -1);
  for (int64_t i = 0; i < n; ++i) {
    mark[i] = (int32_t)i;
    for (int64_t p = rp[i]; p < rp[i + 1]; ++p) {
      int32_t k = ci[p];
      while (k != -1 && mark[k] != i) {
        cc[k]++;
        mark[k] = (int32_t)i;
        k = parent[k];
      }
    }
  }
  // the fill of L itself: what the method needs, before amalgamation pads it
  S.nnz_L_exact = 0;
  for (int64_t j = 0; j < n; ++j) S.nnz_L_exact += cc[j] - 1;
  // supernodes: j joins j-1 when parent[j-1] == j and the structures nest
  S.sup_first.clear();
  for (int64_t j = 0; j < n; ++j) {
    bool start = (j == 0) || parent[j - 1] != j || cc[j - 1] != cc[j] + 1 ||
                 (j - S.sup_first.back()) >= max_width;
    if (start) S.sup_first.push_back((int32_t)j);
  }
  S.nsup = (int32_t)S.sup_first.size();
  S.sup_first.push_back((int32_t)n);
  std::vector<int32_t> col2sup(n);
  for (int32_t s = 0; s < S.nsup; ++s)
    for (int32_t j = S.sup_first[s]; j < S.sup_first[s + 1]; ++j) col2sup[j] = s;
  // row structures: own columns, then A's rows below plus children's rows
  std::vector<std::vector<int32_t>> offrows(S.nsup);
  std::vector<std::vector<int32_t>> kids(S.nsup);
  // column pattern (lower) of A in the final numbering, from the row lists
  std::vector<int64_t> cp(n + 1, 0);
  for (int64_t p = 0; p < rp[n]; ++p) cp[ci[p] + 1]++;
  for (int64_t j = 0; j < n; ++j) cp[j + 1] += cp[j];
  std::vector<int32_t> cr(rp[n]);
  {
    std::vector<int64_t> fill(cp.begin(), cp.end() - 1);
    for (int64_t i = 0; i < n; ++i)
      for (int64_t p = rp[i]; p < rp[i + 1]; ++p) cr[fill[ci[p]]++] = (int32_t)i;
  }
  std::fill(mark.begin(), mark.end(), -1);
  S.sup_parent.assign(S.nsup, -1);
  for (int32_t s = 0; s < S.nsup; ++s) {
    int32_t f = S.sup_first[s], l = S.sup_first[s + 1];
    std::vector<int32_t>& rows = offrows[s];
    for (int32_t j = f; j < l; ++j)
      for (int64_t p = cp[j]; p < cp[j + 1]; ++p) {
        int32_t i = cr[p];
        if (i >= l && mark[i] != s) { mark[i] = s; rows.push_back(i); }
      }
    for (int32_t c : kids[s])
      for (int32_t i : offrows[c])
        if (i >= l && mark[i] != s) { mark[i] = s; rows.push_back(i); }
    std::sort(rows.begin(), rows.end());
    if (!rows.empty()) {
      int32_t par = col2sup[rows[0]];
      S.sup_parent[s] = par;
      kids[par].push_back(s);
    }
    if ((int64_t)rows.size() + (l - f) != cc[f]) return "supernode structure mismatch";
  }
  // Relaxed amalgamation: a supernode joins its parent when it is the parent's
  // last child (adjacent columns) and the explicit zeros of the merged dense
  // block stay small; fewer, wider supernodes mean fewer tree levels and
  // denser panels for the solves.  Thresholds: merged width <= 4 always;
  // <= 16 with < 80% zeros; <= 48 with < 10%; otherwise < 5%.
  std::vector<int64_t> zeros;  // explicit zeros of each supernode's panel
  {
    const int32_t ns = S.nsup;
    std::vector<int32_t> first(ns), last(ns);
    zeros.assign(ns, 0);
    std::vector<char> gone(ns, 0);
    for (int32_t t = 0; t < ns; ++t) {
      first[t] = S.sup_first[t];
      last[t] = S.sup_first[t + 1];
    }
    for (int32_t t = 0; t < ns; ++t) {
      const int32_t par = S.sup_parent[t];
      if (par < 0 || last[t] != first[par]) continue;
      const int64_t ws = last[t] - first[t], wp = last[par] - first[par];
      const int64_t rt = (int64_t)offrows[t].size(), rpar = (int64_t)offrows[par].size();
      const int64_t w = ws + wp;
      if (w > max_width) continue;
      const int64_t z = zeros[t] + zeros[par] + ws * (wp + rpar - rt);
      const double dense = (double)w * (double)(w + 1) / 2.0 + (double)w * (double)rpar;
      const double zf = (double)z / dense;
      const bool merge = w <= 4 || (w <= 16 && zf < 0.8) || (w <= 48 && zf < 0.1) || zf < 0.05;
      if (!merge) continue;
      first[par] = first[t];
      zeros[par] = z;
      gone[t] = 1;
    }
    keep_supernodes(S, offrows, col2sup, zeros, first, gone);
  }
  // The top levels hold few supernodes whose separators are nearly dense in
  // each other: as one supernode of at most kTopWidth columns they cost one
  // launch per direction instead of one each.
  std::vector<int32_t> lev = sup_levels(S);
  const int32_t l0 = top_level(S, lev, std::min<int64_t>({max_width, kTopWidth, n / 8}));
  order_children(S, offrows, col2sup, zeros, lev, l0);
  if (n > kTopMinN) {
    merge_top(S, offrows, col2sup, zeros, lev, l0);
    lev.clear();
  }
  if (coarse) {
    *coarse = S;
    std::vector<std::vector<int32_t>> rows = offrows;
    std::vector<int32_t> c2s = col2sup;
    if (!lev.empty()) merge_top(*coarse, rows, c2s, zeros, lev, l0);
    amalgamate_tiled(*coarse, rows, c2s, zeros, max_width);
    lay_out(*coarse, rows);
  }
  lay_out(S, offrows);
  return "";
}

}  // namespace matex
