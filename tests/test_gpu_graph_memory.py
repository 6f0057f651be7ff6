"""A graph whose bit matrices do not fit in device memory: it is created all
the same, without them, and gives the results of one that has them."""
import pytest

import cudart_shim

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CODE = """
import json, os
import mqo_inputs as mi
import paper_2605_06921_gb300 as mq
import torch
P = mi.pack([mi.erdos_renyi(n, 0.2, n) for n in (300, 130)])
if os.environ.get("FAIL"):
    # 128 columns of a row in 16 bytes, rows in tiles of 128; the tile list: 8 bytes each
    tiles = [(n + 127) // 128 for n in (300, 130)]
    os.environ["SHIM_FAIL_BYTES"] = str({"bits": sum(t * t * 128 * 16 for t in tiles), "tiles": 8 * sum(tiles)}[
        os.environ["FAIL"]])
g = mq.Graph(P)
os.environ.pop("SHIM_FAIL_BYTES", None)
s = mq.Solver(g, mq.params(batch=32, x_dtype=1, t_gs=2, descent_cap=20, seed=3))
assert s.info()["disc_bits"] == (not os.environ.get("FAIL")), s.info()
s.run(60)
s.local_search()
v, bits = s.best()
e = [t.tolist() for t in s.evaluate(bits)]
x = torch.linspace(0, 1, P.n * 32, device="cuda").view(P.n, 32)
print(json.dumps([v.tolist(), bits.tolist(), e, s.traj_state(), mq.spmm_grad(g, x, 0.001).double().sum().item()]))
"""


def test_graph_without_room_for_its_bit_matrices(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    want = cudart_shim.run(tmp_path, CODE)
    for what in ("bits", "tiles"):
        assert cudart_shim.run(tmp_path, CODE, FAIL=what) == want
