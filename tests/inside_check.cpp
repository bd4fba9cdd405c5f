// CPU check of csrc/inet_inside.h: nets reduced with the templates that hold
// reduced pairs must come to the same normal form, with the same number of
// applications of every loaded rule, as with the loaded templates.  A plain
// sequential interpreter of templates; the first line of the output is the
// number of rules with a reduced pair and how often they were applied.
#include <cstdio>
#include <fstream>
#include <sstream>
#include <string>
#include <vector>

#include "inet_inside.h"
#include "inet_text.h"

using namespace inet;

namespace {

std::string slurp(const char* path) {
  std::ifstream f(path);
  std::stringstream s;
  s << f.rdbuf();
  return s.str();
}

struct Machine {
  const CompiledRules& rules;
  const std::vector<Template>& tmpl;
  const std::vector<std::vector<int>>& more;
  std::vector<Node> nodes;
  std::vector<uint32_t> vars;
  std::vector<Pair> todo;
  std::vector<long> hist;
  long inside = 0;

  void link(uint32_t t, uint32_t u) {
    for (;;) {
      if (is_agent(t) && is_agent(u)) {
        todo.push_back({idx_of(t), idx_of(u)});
        return;
      }
      if (!is_var(t)) std::swap(t, u);
      uint32_t& cell = vars[idx_of(t)];
      const uint32_t old = cell;
      cell = u;
      if (old == kEmpty) return;
      cell = kEmpty;
      t = old;
    }
  }
  void run() {
    const int L = rules.n_labels();
    while (!todo.empty()) {
      Pair p = todo.back();
      todo.pop_back();
      const int e = rules.table[(size_t)(nodes[p.a].head & 0xFF) * (size_t)L + (size_t)(nodes[p.b].head & 0xFF)];
      if (e < 0) continue;
      if (e & 1) std::swap(p.a, p.b);
      const size_t ti = (size_t)e >> 1;
      const Template& t = tmpl[ti];
      hist[ti]++;
      for (int r : more[ti]) hist[(size_t)r]++;
      inside += (long)more[ti].size();
      uint32_t v[kNumVals] = {};
      for (int q = 0; q < 3; q++) {
        v[kValExt + q] = nodes[p.a].aux[q];
        v[kValExt + 3 + q] = nodes[p.b].aux[q];
      }
      for (int j = 0; j < t.n_new; j++) {
        v[kValNew + j] = mk_agent((uint32_t)nodes.size());
        nodes.push_back(Node{t.lab[j], {0, 0, 0}});
      }
      for (int f = 0; f < t.n_fresh; f++) {
        v[kValFresh + f] = mk_var((uint32_t)vars.size());
        vars.push_back(kEmpty);
      }
      for (int j = 0; j < t.n_new; j++)
        for (int q = 0; q < 3; q++)
          if (t.src[j][q] != kValNone) nodes[idx_of(v[kValNew + j])].aux[q] = v[t.src[j][q]];
      for (int k = 0; k < t.n_link; k++) link(v[t.link[k][0]], v[t.link[k][1]]);
    }
  }
};

}  // namespace

int main(int argc, char** argv) {
  if (argc < 3) return 2;
  CompiledRules rules;
  std::string err;
  if (compile_rules(slurp(argv[1]), rules, err)) {
    printf("%s\n", err.c_str());
    return 1;
  }
  std::vector<Template> spec;
  std::vector<std::vector<int>> more, none(rules.tmpl.size());
  inside_rules(rules.tmpl.data(), rules.tmpl.size(), &spec, &more);
  int with = 0;
  for (auto& m : more) with += !m.empty();
  long applied = 0;
  std::istringstream nets(slurp(argv[2]));
  for (std::string line; std::getline(nets, line);) {
    std::string text[2];
    std::vector<long> hist[2];
    for (int k = 0; k < 2; k++) {
      FlatNet fn;
      if (flatten_net(line, rules, 0, 0, 0, fn, err)) {
        printf("%s: %s\n", line.c_str(), err.c_str());
        return 1;
      }
      Machine m{rules, k ? spec : rules.tmpl, k ? more : none, fn.nodes, fn.vars, fn.pairs,
                std::vector<long>(rules.tmpl.size())};
      m.run();
      Readback rb;
      read_net(m.nodes.data(), m.nodes.size(), m.vars.data(), m.vars.size(), fn.iface, rules, 1u << 20, true, rb);
      text[k] = rb.text;
      hist[k] = m.hist;
      applied += m.inside;
    }
    if (text[0] != text[1] || hist[0] != hist[1]) {
      printf("%s: %s against %s\n", line.c_str(), text[1].c_str(), text[0].c_str());
      return 1;
    }
  }
  printf("%d %ld\n", with, applied);
  return 0;
}
