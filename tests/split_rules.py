"""The host rules that split a sweep into CTAs (csrc/mfc_launch.cuh), restated; the
functions of the header are compiled and compared with these in test_split_rules.py."""
import os
import re
import subprocess

LAUNCH = os.path.join(os.path.dirname(os.path.abspath(__file__)), os.pardir, "paper_2305_09163_gb300", "csrc",
                      "mfc_launch.cuh")


def chunks_per_block(slots):
    """Chunks of 128 slots that one x CTA walks (it finishes 128 k - 2)."""
    return min(max((slots + 125) // 126 // (152 * 16), 1), 16)


def segment(plane, n, fp64):
    """Cells per segment of a y/z sweep."""
    columns, tail = (plane + 31) // 32, 1.0 if fp64 else 2.5
    best = least = None
    for L in range(2, n + 4, 4):
        walk = (L + 2) // 4 + 0.25
        t = (n // L * walk + ((n % L + 5) // 4 + 0.25 if n % L else 0.0)) * columns / 152.0 + tail * walk
        if least is None or t < least:
            best, least = L, t
        if L >= n:
            break
    return best


def compile_rules(out_dir):
    with open(LAUNCH) as f:
        src = f.read()
    parts = [m.group(0) for m in re.finditer(r"^constexpr long long kStream\w+ = [^;]*;", src, re.M)]
    parts += [re.search(r"inline \w+(?: long)? %s\(.*?\n}\n" % fn, src, re.S).group(0)
              for fn in ("stream_slots_per_block", "stream_segment")]
    cpp, so = os.path.join(out_dir, "rules.cpp"), os.path.join(out_dir, "rules.so")
    with open(cpp, "w") as f:
        f.write("constexpr int kStreamThreads = 128;\n" + "\n".join(parts) + """
extern "C" {
long long slots(long long total) { return stream_slots_per_block(total); }
int segment(long long cells, int n, int fp64) { return stream_segment(cells, n, fp64 != 0); }
}
""")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", cpp, "-o", so], check=True)
    return so
