"""The rule the row kernels' early loads rest on: a kernel that lets its successor start early has first waited for
its predecessor, so whatever a launch reads before its own wait was final two launches ago.  Every kernel that is
launched with programmatic serialisation begins with pdl_enter(), which waits and then releases, and nothing else in
the sources releases a successor."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_05647_gb300", "csrc")
SRC = {os.path.basename(p): open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu*"))}


def test_only_pdl_enter_releases_and_it_waits_first():
    at = {f: t.count("griddepcontrol.launch_dependents") for f, t in SRC.items()}
    assert {f for f, n in at.items() if n} == {"internal.cuh"} and at["internal.cuh"] == 1
    body = re.search(r"void pdl_enter\(\)\s*\{(.*?)\n\}", SRC["internal.cuh"], re.S).group(1)
    assert body.index("griddepcontrol.wait") < body.index("griddepcontrol.launch_dependents")


def _kernels():
    """name -> body of every __global__ function."""
    out = {}
    for t in SRC.values():
        for m in re.finditer(r"__global__", t):
            sig = re.compile(r"\b(k_\w+)\s*\(").search(t, m.end())
            i = t.index("\n{", sig.end())
            out[sig.group(1)] = t[i:t.index("\n}", i)]
    return out


def test_every_early_launched_kernel_waits():
    kernels = _kernels()
    launched = set()
    for t in SRC.values():
        for m in re.finditer(r"launch_pdl\(\s*(k_\w+|kern)\b", t):
            if m.group(1) == "kern":
                launched |= set(re.findall(r"\bk_\w+", re.findall(r"auto kern = ([^;]*);", t[:m.start()])[-1]))
            else:
                launched.add(m.group(1))
    assert {"k_kinetic", "k_h2d", "k_e3d", "k_eh2d_v4", "k_copy", "k_kinetic_nl_walk", "k_mlp_train_tile1"} <= launched
    for name in launched:
        body = kernels[name]
        assert "pdl_enter()" in body, name
        # no block leaves before it: an early exit would count as a release
        assert "return;" not in body[:body.index("pdl_enter()")], name
