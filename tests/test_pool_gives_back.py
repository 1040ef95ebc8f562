"""Device memory that the library keeps unused between calls is given back when one of
its own allocations would fail without it (a limit on a stand-in device): a tree's
copies, the rank predictor's buffers, pinned memory aside."""

import fake_runtime

SCRIPT = r"""
from paper_1905_10602_gb300.workloads import bumpy_sphere
MB = 1 << 20
def tree(n):
    t = ifmm.ifmm_build_tree(bumpy_sphere(n, 1), 4)
    ifmm.ifmm_color(t, 3)
    return t
n = 20000
a = tree(n)
ifmm.bem_matvec(a, np.ones(n), kernel=ifmm.default_kernel(n, "df"))  # 25 MB of partial sums, kept afterwards
kept = fake.fake_in_use(0)
assert kept > 25 * MB
fake.fake_limit(0, kept)
b = tree(4000)
ifmm.bem_matvec(b, np.ones(4000))
assert fake.fake_in_use(0) < kept
fake.fake_limit(0, 1000 * MB)
ifmm.bem_matvec(a, np.ones(n), kernel=ifmm.default_kernel(n, "df"))
fake.fake_limit(0, fake.fake_in_use(0))
w = np.zeros(9025, np.float32)
ifmm.ifmm_mlp_forward(w, np.zeros((50000, 9), np.float32))
ifmm.ifmm_mlp_grad(w, np.zeros((50000, 9), np.float32), np.zeros(50000, np.float32))
# what is in use is not given away
fake.fake_limit(0, 1)
try:
    t = tree(5000)
    ifmm.bem_matvec(t, np.ones(5000))
    assert False
except ifmm.IFMMError as e:
    assert "IFMM_ENOMEM" in str(e), e
"""


def test_pool_gives_back(tmp_path):
    fake_runtime.run(SCRIPT, tmp_path)
