"""The FP64 products' buffers (digit images of the tensor, the product) are an addition: on a device
that is nearly full a handle does without them, so that its create, its gradients, a run with
compaction and the standard errors find the memory they need, and gives what the CUDA-core kernel
gives, bit for bit.  In a process of its own: memory freed by earlier handles stays in the library's
pool."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = """
import numpy as np, torch
from paper_2112_03985_gb300 import api
dims, R = (150, 100, 50), 5                  # images and product: about 150 MB
rng = np.random.default_rng(0)
T = rng.random(dims)
U = [rng.random((I, 150 * R)) for I in dims]
left = [[p] for p in range(150)]
ref = api.JKCALS(T, 0, [R] * 150, left, U, max_device_bytes=1 << 46)
full = api.JKCALS(T, 0, [R] * 150, left, U)
want, other = ref.mttkrp(1), full.mttkrp(1)
assert (np.asarray(want) != np.asarray(other)).any(), "with room the size takes the products"
grad = ref.grad()
ref.run(20, 1e-3)
se = ref.jackknife_se(ref_block=0)
ref.close(); full.close()
torch.cuda.synchronize()
# {free} MB beside what the library's pool still holds
room = {free} << 20
hs = []
free, _ = torch.cuda.mem_get_info()
fill = torch.empty(free - room, dtype=torch.uint8, device="cuda")
# use up what the pool kept: handles until one does not take the products
for k in range(12):
    h = api.JKCALS(T, 0, [R] * 150, left, U)
    hs.append(h)
    if (np.asarray(h.mttkrp(1)) == np.asarray(want)).all():
        break
else:
    raise AssertionError("twelve handles took the products")
# the handle without them does everything
g = h.grad()
assert g[0] == grad[0] and all((np.asarray(a) == np.asarray(b)).all() for a, b in zip(g[1], grad[1]))
h.run(20, 1e-3)
s = h.jackknife_se(ref_block=0)
for a, b in zip(s[0], se[0]):
    if a is not None:
        assert (a == b).all()
# and so do those before it
for x in hs[:-1]:
    x.grad(); x.run(20, 1e-3); x.jackknife_se(ref_block=0)
print("handles", len(hs))
"""


@pytest.mark.parametrize("free", [1200])
def test_a_nearly_full_device(free):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", SCRIPT.replace("{free}", str(free))], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
