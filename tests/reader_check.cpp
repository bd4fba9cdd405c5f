// CPU check of the two net readers of csrc/inet_text.cpp: PlainReader must take
// exactly the texts that NetReader accepts, with the same records, name slots,
// interface and pairs.  Texts: random nets of up to 400 names (around the
// number from which names are hashed, too) with comments and blanks anywhere,
// and random edits of them.  Prints how many texts were accepted and refused.
#include "inet_text.cpp"

#include <random>

using namespace inet;

namespace {

std::mt19937_64 rng(14040076);
uint32_t pick(uint32_t n) { return (uint32_t)(rng() % n); }

const char* const kRules =
    "Add(y, r) = Z -> r = y;\nAdd(y, r) = S(x) -> Add(y, w) = x, r = S(w);\n"
    "Dup(a, b) = Z -> a = Z, b = Z;\nDup(a, b) = S(x) -> Dup(p, q) = x, a = S(p), b = S(q);\n"
    "Tri(a, b, c) = Nil_0' -> a = b, c = Z;\n";

// Something between two tokens: nothing, blanks, or a comment.
std::string gap() {
  switch (pick(12)) {
    case 0: return " ";
    case 1: return "\n\t";
    case 2: return "  \r\n";
    case 3: return "# a comment < | >, x = y (\n";
    case 4: return "#\n #x\n";
    default: return "";
  }
}

struct Gen {
  std::vector<std::string> open;  // names that occurred once
  int made = 0, most;
  explicit Gen(int m) : most(m) {}
  std::string fresh() {
    static const char* const stem[] = {"x", "y", "z_", "name", "aVeryLongNameIndeed", "q'"};
    std::string n = stem[pick(6)] + std::to_string(made++);
    open.push_back(n);
    return n;
  }
  std::string name() {
    if (!open.empty() && (made >= most || pick(2))) {
      const size_t k = pick((uint32_t)open.size());
      std::string n = open[k];
      open.erase(open.begin() + (long)k);
      return n;
    }
    return made < most ? fresh() : std::string("Z");
  }
  std::string term(int depth) {
    if (depth == 0 || pick(3) == 0) return pick(2) ? name() : std::string(pick(2) ? "Z" : "Nil_0'");
    static const struct { const char* sym; int ar; } kSym[] = {{"S", 1}, {"Add", 2}, {"Dup", 2}, {"Tri", 3}, {"Z", 0}};
    const auto& s = kSym[pick(5)];
    std::string t = s.sym + gap();
    if (s.ar == 0) return pick(3) ? t : t + "(" + gap() + ")";
    t += "(" + gap();
    for (int i = 0; i < s.ar; i++) t += (i ? "," + gap() : "") + term(depth - 1) + gap();
    return t + ")";
  }
  std::string net(int eqs) {
    std::string t = gap() + "<" + gap();
    const int roots = (int)pick(4);
    for (int i = 0; i < roots; i++) t += (i ? "," + gap() : "") + term(2) + gap();
    t += "|" + gap();
    for (int i = 0; i < eqs; i++) t += (i ? "," + gap() : "") + term((int)pick(4)) + gap() + "=" + gap() + term((int)pick(4)) + gap();
    return t + ">" + gap() + (pick(8) ? "" : "# to the end");
  }
};

bool equal(const FlatNet& a, const FlatNet& b) {
  return a.vars == b.vars && a.iface == b.iface && a.nodes.size() == b.nodes.size() && a.pairs.size() == b.pairs.size() &&
         (a.nodes.empty() || memcmp(a.nodes.data(), b.nodes.data(), a.nodes.size() * sizeof(Node)) == 0) &&
         (a.pairs.empty() || memcmp(a.pairs.data(), b.pairs.data(), a.pairs.size() * sizeof(Pair)) == 0);
}

}  // namespace

int main() {
  CompiledRules rules;
  std::string err;
  if (compile_rules(kRules, rules, err)) return printf("%s\n", err.c_str()), 1;
  int taken = 0, refused = 0;
  for (int i = 0; i < 6000; i++) {
    const int names = i % 3 == 0 ? (int)pick(6) : i % 3 == 1 ? 14 + (int)pick(6) : (int)pick(400);
    std::string t = Gen(names).net((int)pick(3) + names / 2);
    if (i % 2) {  // an edit, mostly an error
      const size_t at = pick((uint32_t)t.size() + 1);
      const char c = "(),=|<>;xyzSZ -#\n\0"[pick(18)];
      if (pick(2)) t.insert(at, 1, c);
      else if (at < t.size()) t.erase(at, 1 + pick(3));
    }
    const uint32_t ab = pick(1000), vb = pick(1000), slot = pick(100);
    FlatNet a, b;
    std::string e;
    const bool plain = PlainReader{rules, slot, ab, vb, a}.net(t);
    const bool full = NetReader{t, rules, slot, ab, vb, b, e}.net();
    if (plain != full || (full && !equal(a, b)))
      return printf("%s: plain reader %d, full reader %d (%s)\n", t.c_str(), plain, full, e.c_str()), 1;
    (full ? taken : refused)++;
  }
  printf("%d %d\n", taken, refused);
  return 0;
}
