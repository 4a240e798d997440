"""The lattice tuner times each launch shape once.  Strips hold at most 16 words,
so two candidates with the same threads a block and lanes are one shape.  (Read
from the source: the list of candidates is not part of the interface.)"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_candidates_differ():
    text = open(os.path.join(ROOT, "paper_1811_04384_gb300", "csrc", "ising_tune.cu")).read()
    cands = re.search(r"std::vector<Candidate> cands = \{(.*?)\};", text, re.S).group(1)
    shapes = [(int(bg) if bw == "0" else int(bw) * int(bg), path, lanes)
              for bw, bg, path, lanes in re.findall(r"\{(\d+), (\d+), (\w+), (\d+)\}", cands)]
    assert len(shapes) == len(set(shapes)) and len(shapes) >= 9
    assert {t for t, path, lanes in shapes if path == "P" and lanes == "1"} == {32, 64, 128, 192, 256}
