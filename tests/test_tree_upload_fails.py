"""A tree whose device copies fail half-way for want of memory (a limit on a stand-in
device) has none of them afterwards: the next call makes them all, instead of taking
the first for the whole."""

import fake_runtime

SCRIPT = r"""
from paper_1905_10602_gb300.workloads import bumpy_sphere
n = 20000
t = ifmm.ifmm_build_tree(bumpy_sphere(n, 1), 4)
ifmm.ifmm_color(t, 3)
for room in (24 * n + 8, 28 * n + 8):  # the points; the points and the permutation
    fake.fake_limit(0, room)
    try:
        ifmm.bem_matvec(t, np.ones(n))
        assert False
    except ifmm.IFMMError as e:
        assert "IFMM_ENOMEM" in str(e), e
    assert fake.fake_in_use(0) == 0
fake.fake_limit(0, 1 << 30)
ifmm.bem_matvec(t, np.ones(n))
assert fake.fake_in_use(0) >= 52 * n
"""


def test_all_copies_or_none(tmp_path):
    fake_runtime.run(SCRIPT, tmp_path)
