"""The net reader for well-formed texts (csrc/inet_text.cpp, PlainReader) takes
every text that the full reader accepts, nets of many names and texts with
comments among them, and reads the same net from it (CPU)."""
import os
import subprocess

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
