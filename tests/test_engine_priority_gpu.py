"""An engine's groups run as graph branches at the priority of the engine's stream:
the priorities of the captured kernels, read from the graph as it is
instantiated (a preloaded wrapper, in a process of its own)."""
import os
import shutil
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
RUN = """
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_2005_13425_gb300 import inputs, nekgb as nek
stream = torch.cuda.Stream(priority=-1)
torch.cuda.set_stream(stream)
eng = nek.nb_engine_create(256 << 20, stream)
for n in (4, 6, 8):
    f = torch.from_numpy(inputs.unique_field(2, 2, 2, n, seed=n)).cuda()
    nek.nb_engine_submit_unique(eng, (2, 2, 2), n, inputs.PERTURB_AMP, (0.3, -0.5, 0.7), 0.0, 16, f)
print("stream", stream.priority, flush=True)
nek.nb_engine_step(eng, 8)
stream.synchronize()
nek.nb_engine_destroy(eng)
"""


def test_branches_keep_the_streams_priority(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_13425_gb300 import build as b
    b.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    shim = str(tmp_path / "graph_priorities.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "host", "graph_priorities.cpp"), "-o", shim, "-ldl"], check=True)
    # the tuner's choices, so that only the step's own graph is captured
    tune = tmp_path / "tune"
    p = torch.cuda.get_device_properties(0)
    tune.write_text("".join("n%d_fp64_sm%d_%s 1 8\n" % (n, p.multi_processor_count, p.name.replace(" ", "_"))
                            for n in (4, 6, 8)))
    env = dict(os.environ, LD_PRELOAD=shim, NEKGB_TUNE_CACHE=str(tune))
    out = subprocess.run([sys.executable, "-c", RUN, os.path.dirname(HERE)], env=env, check=True, capture_output=True,
                         text=True, timeout=300).stdout.splitlines()
    at = out.index("stream -1")
    got = [int(line.split()[-1]) for line in out[at:] if line.startswith("kernel priority")]
    # three groups, each with its own branch; the driver's value of the stream's priority
    assert len(got) >= 3 * 2 * 8 and set(got) == {-1}
