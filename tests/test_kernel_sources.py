"""Ordering that no run on a GPU can show to be missing: what a kernel's source
has to say before it touches memory that others write."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_13903_gb300", "csrc")


def kernels():
    """(file, name, parameters, body) of every __global__ function."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\b", text):
            name = re.compile(r"\b(k_\w+)\s*\(").search(text, m.end())
            ends = [name.end()]
            for open_, close in ("()", "{}"):  # the parameters, then the body
                depth, q = (1, ends[-1]) if open_ == "(" else (0, ends[-1])
                while True:
                    depth += (text[q] == open_) - (text[q] == close)
                    q += 1
                    if depth == 0 and text[q - 1] == close:
                        break
                ends.append(q)
            out.append((os.path.basename(path), name[1], text[ends[0]:ends[1] - 1],
                        text[ends[1]:ends[2]]))
    return out


def test_a_cluster_meets_before_it_stores_into_its_ctas():
    """Distributed shared memory belongs to a CTA that has started: a barrier of
    the whole cluster comes before the programs that store into it."""
    body = {k[1]: k[3] for k in kernels()}["k_coarse"]
    assert 0 <= body.find("barrier_arrive(") < body.find("barrier_wait(") < body.find("p.run_")


def test_inputs_of_early_placed_kernels_are_not_read_as_constant():
    """A kernel placed while its predecessor still writes must not promise that
    its inputs stay as they are from the launch on (const T* __restrict__)."""
    early = [k for k in kernels() if "after_previous(" in k[3]]
    assert len(early) > 40
    for file, name, params, _ in early:
        for p in params.split(","):
            assert not ("const" in p and "__restrict__" in p), (file, name, p.strip())
