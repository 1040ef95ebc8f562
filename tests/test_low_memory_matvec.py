"""The float-pair products with too little memory for the symmetric kernel's partial
sums (a limit on a stand-in device): they take the full sums, which need none, and
nothing of that is remembered for a call with room."""

import fake_runtime

SCRIPT = r"""
from paper_1905_10602_gb300.workloads import bumpy_sphere
n = 20000  # partial sums: 157 tiles x 20,000 x 8 bytes = 25 MB; the product's vectors 0.6 MB
pts = bumpy_sphere(n, 1)
x = np.ones(n)
k = ifmm.default_kernel(n, "df")
def tree():
    t = ifmm.ifmm_build_tree(pts, 4)
    ifmm.ifmm_color(t, 3)
    return t
def block(t):
    return list(ifmm.ifmm_tree_query(t, 0, "matvec_block"))
def product(t):
    fake.fake_clear()
    ifmm.bem_matvec(t, x, kernel=k)
    return launches("k_matvec_df"), launches("k_matvec_symILi")
MB = 1 << 20
fake.fake_limit(0, 10 * MB)
t = tree()
full, sym = product(t)
assert full > 0 and sym == 0, (full, sym)
assert product(t) == (1, 0)  # the choice among the full sums is made once
assert block(t) == [0, 0]
try:
    ifmm.bem_gmres(t, x, kernel=k, restart=5)
except ifmm.IFMMError as e:
    assert "b is zero" in str(e), e  # (the stand-in's kernels compute nothing)
fake.fake_limit(0, 1000 * MB)
full, sym = product(t)
assert full == 0 and sym > 0, (full, sym)
assert block(t)[1] == 3
assert product(t) == (0, 1)
# the same with a size whose symmetric tile is known already (the last tree's end trims the pool)
del t
fake.fake_limit(0, 10 * MB)
t = tree()
assert product(t) == (1, 0)
fake.fake_limit(0, 1000 * MB)
assert product(t) == (0, 1)
"""


def test_full_sums_when_short_of_memory(tmp_path):
    fake_runtime.run(SCRIPT, tmp_path)


FULL64 = r"""
from paper_1905_10602_gb300.workloads import bumpy_sphere
n = 3000
t = ifmm.ifmm_build_tree(bumpy_sphere(n, 1), 3)
ifmm.ifmm_color(t, 3)
for k, x, name in ((ifmm.default_kernel(n), np.ones(n), "8k_matvecE"),
                   (ifmm.helmholtz_kernel(n, 5.0), np.ones(n, complex), "10k_matvec_cE")):
    fake.fake_clear()
    ifmm.bem_matvec(t, x, kernel=k)
    assert launches(name) == 1 and launches("k_matvec64_sym") == 0
"""


def test_switch_to_the_fp64_full_sums(tmp_path):
    fake_runtime.run(FULL64, tmp_path, {"IFMM_MATVEC64_FULL": "1"})
