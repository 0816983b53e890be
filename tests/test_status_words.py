"""Calls of entry points without a context hold a status word each: none is shared by two calls in flight,
and no other word of that kind exists in the library's sources."""
import re
import subprocess
from pathlib import Path

ROOT = Path(__file__).resolve().parents[1]
CSRC = ROOT / "paper_2301_04259_gb300" / "csrc"


def test_no_word_has_two_holders(tmp_path):
    exe = tmp_path / "words"
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", f"-I{CSRC}", str(ROOT / "tests/native/status_words.cpp"),
                    "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.split()[0] == "0", r.stdout


def test_no_single_status_word_is_left():
    words = [m for f in sorted(CSRC.glob("*.cu")) for m in
             re.findall(r"static __device__ unsigned int (\w+(?:\[\w+\])?);", f.read_text())]
    assert words == ["g_call_words[kCallWords]"]
