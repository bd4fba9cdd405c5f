// Active pairs inside a right-hand side, reduced when the rules are compiled:
// a rule whose right-hand side joins two of its own new agents principal port
// to principal port (Fib2(r) = S(x) -> .., Fib(w1) = S(a)) is always followed
// by the rule of that pair, so the specialised kernel applies both as one.
// One interaction fewer on every path through such a rule, and two agents
// that are never written: Ackermann(3, 4..8) 68 -> 45 ms together with the
// runs it makes possible (inet_async.cuh).
// Plain C++17; no CUDA.
#pragma once

#include <cstddef>
#include <cstring>
#include <vector>

#include "inet_layout.h"

namespace inet {

// Wires of a right-hand side: the partner of each terminal.  Terminals: the
// left-hand side's arguments E(e) = e (0..5), then the principal port
// 6 + 4 j and the auxiliary ports 6 + 4 j + 1 + p of new agent j.
inline int term_of(int code) { return code < kValNew ? code : 6 + 4 * (code - kValNew); }

inline std::vector<int> wires(const Template& t) {
  std::vector<int> par(6 + 4 * (size_t)t.n_new, -1);
  std::vector<int> seen(kMaxFresh, -1);
  auto join = [&](int a, int b) { par[(size_t)a] = b; par[(size_t)b] = a; };
  for (int j = 0; j < t.n_new; j++)
    for (int p = 0; p < 3; p++) {
      const int c = t.src[j][p], x = 6 + 4 * j + 1 + p;
      if (c == kValNone) continue;
      if (c < kValFresh) join(x, term_of(c));
      else if (seen[(size_t)(c - kValFresh)] < 0) seen[(size_t)(c - kValFresh)] = x;
      else join(x, seen[(size_t)(c - kValFresh)]);
    }
  for (int k = 0; k < t.n_link; k++) join(term_of(t.link[k][0]), term_of(t.link[k][1]));
  return par;
}

// Rule r with the active pair of its new agents j1 and j2 reduced by rule s
// (Sec. 2.2: ->int on a pair both of whose agents the rule itself creates,
// so it is the next interaction whatever the rest of the net does).  `swap`:
// j1 is the second symbol of s's left-hand side.  False when the result does
// not fit a template.
inline bool reduce_inside(const Template& r, const Template& s, int j1, int j2, bool swap, Template* out) {
  const std::vector<int> pr = wires(r), ps = wires(s);
  const int side[2] = {swap ? j2 : j1, swap ? j1 : j2};  // s's alpha and beta
  const int nr = r.n_new, ns = s.n_new;
  if (nr - 2 + ns > kMaxNew) return false;
  std::vector<int> at((size_t)nr, -1);  // r's agents in the result, then s's
  int n = 0;
  for (int j = 0; j < nr; j++)
    if (j != j1 && j != j2) at[(size_t)j] = n++;
  const int base = n;
  n += ns;
  auto inner = [&](int t) { return t >= 6 && ((t - 6) / 4 == j1 || (t - 6) / 4 == j2); };
  // the result's terminal for r's / s's
  auto of_r = [&](int t) { return t < 6 ? t : 6 + 4 * at[(size_t)((t - 6) / 4)] + (t - 6) % 4; };
  auto of_s = [&](int t) { return 6 + 4 * (base + (t - 6) / 4) + (t - 6) % 4; };
  auto arg_of = [&](int t) { return ((t - 6) / 4 == side[0] ? 0 : 3) + (t - 6) % 4 - 1; };  // r's inner port as s's argument
  auto port_of = [&](int e) { return 6 + 4 * side[e / 3] + 1 + e % 3; };
  // where a wire that enters r's terminal u ends
  auto end = [&](int u, bool in_r) -> int {
    for (int guard = 0; guard < 64; guard++) {
      if (u < 0) return -1;
      if (in_r) {
        if (!inner(u)) return of_r(u);
        if ((u - 6) % 4 == 0) return -1;
        u = ps[(size_t)arg_of(u)];
        in_r = false;
      } else {
        if (u >= 6) return of_s(u);
        u = pr[(size_t)port_of(u)];
        in_r = true;
      }
    }
    return -1;
  };
  std::vector<int> par(6 + 4 * (size_t)n, -1);
  for (int t = 0; t < (int)pr.size(); t++)
    if (pr[(size_t)t] >= 0 && !inner(t)) {
      if ((par[(size_t)of_r(t)] = end(pr[(size_t)t], true)) < 0) return false;
    }
  for (int t = 6; t < (int)ps.size(); t++)
    if (ps[(size_t)t] >= 0) {
      if ((par[(size_t)of_s(t)] = end(ps[(size_t)t], false)) < 0) return false;
    }
  Template o;
  memset(&o, 0, sizeof o);
  memset(o.src, kValNone, sizeof o.src);
  memset(o.link, kValNone, sizeof o.link);
  o.rule = r.rule;
  o.lhs[0] = r.lhs[0];
  o.lhs[1] = r.lhs[1];
  o.n_new = (uint8_t)n;
  for (int j = 0; j < nr; j++)
    if (at[(size_t)j] >= 0) o.lab[at[(size_t)j]] = r.lab[j];
  for (int j = 0; j < ns; j++) o.lab[base + j] = s.lab[j];
  auto aux = [](int t) { return t >= 6 && (t - 6) % 4 != 0; };
  auto code = [](int t) { return (uint8_t)(t < 6 ? t : kValNew + (t - 6) / 4); };
  for (int t = 0; t < (int)par.size(); t++) {
    const int u = par[(size_t)t];
    if (u < 0 || u < t) continue;
    if (par[(size_t)u] != t) return false;
    if (aux(t) && aux(u)) {
      if (o.n_fresh >= kMaxFresh) return false;
      const uint8_t f = (uint8_t)(kValFresh + o.n_fresh++);
      o.src[(t - 6) / 4][(t - 6) % 4 - 1] = f;
      o.src[(u - 6) / 4][(u - 6) % 4 - 1] = f;
    } else if (aux(t) || aux(u)) {
      const int x = aux(t) ? t : u, y = aux(t) ? u : t;
      o.src[(x - 6) / 4][(x - 6) % 4 - 1] = code(y);
    } else {
      if (o.n_link >= kMaxLink) return false;
      o.link[o.n_link][0] = code(t);
      o.link[o.n_link][1] = code(u);
      o.n_link++;
    }
  }
  *out = o;
  return true;
}

// The rules as the specialised kernel reduces them: each of the first
// kSpecialised (the ones with their own code) with up to kMaxInside of the active pairs that its right-hand
// side itself contains already reduced (Fib2(r) = S(x) -> .., Fib(w1) = S(a)
// goes on to Fib2(w1) = a at once).  `more` lists the rules applied inside.
constexpr size_t kSpecialised = 32;
constexpr int kMaxInside = 2;
inline void inside_rules(const Template* t, size_t n, std::vector<Template>* out, std::vector<std::vector<int>>* more) {
  out->assign(t, t + n);
  more->assign(n, {});
  for (size_t i = 0; i < n && i < kSpecialised; i++) {
    for (int round = 0; round < kMaxInside; round++) {
      Template& r = (*out)[i];
      bool done = false;
      for (int k = 0; k < r.n_link && !done; k++) {
        const int a = r.link[k][0], b = r.link[k][1];
        if (a < kValNew || b < kValNew) continue;
        const int j1 = a - kValNew, j2 = b - kValNew;
        for (size_t s = 0; s < n && !done; s++) {
          const bool fwd = t[s].lhs[0] == r.lab[j1] && t[s].lhs[1] == r.lab[j2];
          const bool rev = t[s].lhs[1] == r.lab[j1] && t[s].lhs[0] == r.lab[j2];
          if (!fwd && !rev) continue;
          Template o;
          if (!reduce_inside(r, t[s], j1, j2, rev, &o)) continue;
          r = o;
          (*more)[i].push_back((int)s);
          done = true;
        }
      }
      if (!done) break;
    }
  }
}

}  // namespace inet
