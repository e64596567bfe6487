"""pgm_check_desc states the memory a built graph holds: within the arrays' alignment (256 bytes each)
and the group records, also where a graph carries the plan of a one-launch run or the blocks of the
fused K-state form; and it asks no device for it."""
import json
import os
import subprocess
import sys

import pytest

from paper_2202_04110_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GRAPHS = {"ising 10x10": lambda: W.ising_grid(10, 10, 0), "ising 20x35": lambda: W.ising_grid(20, 35, 0),
          "ising 317x241": lambda: W.ising_grid(317, 241, 0), "ising 1250x1250": lambda: W.ising_grid(1250, 1250, 0),
          "potts 512 K4": lambda: W.potts_grid(512, 4, 0), "potts 300 K8": lambda: W.potts_grid(300, 8, 0),
          "potts 181 K16": lambda: W.potts_grid(181, 16, 0), "potts 400 K16": lambda: W.potts_grid(400, 16, 0),
          "rbm 300x200": lambda: W.rbm(300, 200, 0), "pool 40": lambda: W.pool_grid(40, 2, 1, 0)}

# the sizes, in a process that sees no device
HOST = ("import json, sys; sys.path.insert(0, {root!r}); from tests.test_gpu_device_bytes import GRAPHS; "
        "from paper_2202_04110_gb300 import binding as B; "
        "print(json.dumps({{k: B.check_desc(f().graph)['device_bytes'] for k, f in GRAPHS.items()}}))")


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_04110_gb300 import build
    build.build()
    from paper_2202_04110_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def host_sizes(gpu):
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")
    out = subprocess.run([sys.executable, "-c", HOST.format(root=ROOT)], env=env, capture_output=True, text=True, check=True, cwd=ROOT)
    return json.loads(out.stdout.splitlines()[-1])


@pytest.mark.parametrize("name", list(GRAPHS))
def test_stated_and_held(gpu, host_sizes, name):
    fg = GRAPHS[name]().graph
    stated = gpu.check_desc(fg)["device_bytes"]
    held = gpu.Graph(fg).info["device_bytes"]
    records = 32 * 256 + 8 * 1024 * (len(fg.enum_groups) + len(fg.logic_groups))
    assert 0 <= held - stated <= records, (stated, held)
    assert host_sizes[name] == stated
