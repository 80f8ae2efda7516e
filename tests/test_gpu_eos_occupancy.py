"""The equation-of-state kernels' block size of a launch follows from the state's species count and the rows
alone, not from the states made before: 17 and 32 species share a kernel instance, but the 64-thread blocks of
17 need half the shared memory, so that more of them fit. Each order in a process of its own; the launches are
read from a captured step."""
import os
import re
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = """
import re, sys, tempfile, os
import torch, synth
import paper_2508_18969_gb300 as df
def step(n, N):
    mech, net = synth.mechanism.make_mechanism(n, 1, 3), synth.network.make_network([n + 2, 32, n], n, seed=1)
    cells = [torch.tensor(a, device="cuda") for a in synth.fields.training_states(mech, N, 5)[:3]]
    st = df.State(mech, net, T_react=0.0, batch_cells=N)
    st.chem_step(*cells)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph):
        st.chem_step(*cells)
    path = os.path.join(tempfile.mkdtemp(), "step.dot")
    graph.debug_dump(path)
    found = re.findall(r"(eos_(?:pre|post)_kernel)[^\\\\]*[\\\\<]+(\\d+),(\\d+),", open(path).read())
    st.close()
    return sorted(found)
for n in map(int, sys.argv[1:]):
    print(n, [step(n, N) for N in (20011, 60013, 77003, 90007)])
"""


def _run(*order):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT, *map(str, order)], cwd=root, capture_output=True, text=True,
                       env={**os.environ, "PYTHONPATH": root}, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return dict(re.findall(r"^(\d+) (.*)$", r.stdout, re.M))


def test_blocks_do_not_depend_on_earlier_states():
    import __graft_entry__ as g
    g.build()
    alone = {**_run(17), **_run(32)}
    assert "'64')" in alone["32"] and "'256')" in alone["32"] and "eos_post" in alone["17"], alone
    assert alone["17"] != alone["32"]
    assert _run(17, 32) == alone and _run(32, 17) == alone
