"""The net reader for well-formed texts (csrc/inet_text.cpp, PlainReader) takes
every text that the full reader accepts, nets of many names and texts with
comments among them, and reads the same net from it (CPU)."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_readers_agree(tmp_path):
    exe = str(tmp_path / "reader_check")
    csrc = os.path.join(ROOT, "paper_1404_0076_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", csrc,
                    os.path.join(ROOT, "tests", "reader_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr
    taken, refused = map(int, r.stdout.split())
    assert taken > 3000 and refused > 1000


def test_a_large_net_leaves_no_large_work_space(tmp_path):
    # what a thread keeps after it has read a large net, and after a large text
    # that is no net at all, does not grow with the text
    code = """
import gc, os, sys
from paper_1404_0076_gb300 import capi as C
def rss():
    gc.collect()
    with open("/proc/self/statm") as f:
        return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")
ctx = C.inet_create(-1)
C.inet_load_rules(ctx, "Add(y, r) = Z -> r = y;\\nAdd(y, r) = S(x) -> Add(y, w) = x, r = S(w);\\n")
C.inet_parsed_free(C.inet_parse_nets(ctx, ["< r | Add(Z, r) = S(Z) >"] * 64))
before = rss()
for text in ("< " + "S(" * 3000000 + "Z" + ")" * 3000000 + " | >", "< | " + ", ".join("n%d = Z" % i for i in range(500000)) + " >",
             "< " + "S(" * 3000000):
    C.inet_parsed_free(C.inet_parse_nets(ctx, [text]))
    del text
print(rss() - before)
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, MALLOC_MMAP_THRESHOLD_=str(1 << 20)))
    assert r.returncode == 0, r.stderr
    assert int(r.stdout) < 24 << 20, r.stdout   # the nets took 100 to 250 MB while they were read
