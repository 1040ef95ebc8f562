"""A process that goes on to a second GPU: function attributes and what was probed
of a kernel's residency belong to a device.  The library's host code runs against two
stand-in devices, the second one without room for clusters of 16 CTAs; every launch
must be one that the runtime would accept there."""

import kernel_calls
import fake_runtime

SCRIPT = r"""
from paper_1905_10602_gb300.workloads import bumpy_sphere
kc = ctypes.CDLL({kc!r})
vp = lambda a: a.ctypes.data_as(ctypes.c_void_p)
w = np.zeros(9025, np.float32)
x, t = np.zeros((100, 9), np.float32), np.zeros(100, np.float32)
pts = bumpy_sphere(700, 3)
fake.fake_max_cluster(1, 8)

def factor(prec):
    tree = ifmm.ifmm_build_tree(pts, 3)
    ifmm.ifmm_color(tree, 3)
    ifmm.ifmm_factor(tree, 4, 1e-6, precision=prec)

def svd(prec, n):
    A, V, sig = np.zeros((n, n)), np.zeros((n, n)), np.zeros(n)
    assert kc.kc_svd(prec, n, vp(A), vp(V), vp(sig)) == 0

def top(n):
    A, X, info = np.zeros((n, n)), np.zeros((n, n)), np.zeros(1, np.int32)
    assert kc.kc_top_inverse(n, vp(A), vp(X), vp(info), 0) == 0

calls = [
    lambda: ifmm.ifmm_mlp_forward(w, x),
    lambda: ifmm.ifmm_mlp_grad(w, x, t),
    lambda: ifmm.ifmm_mlp_train(x, t, epochs=1, batch=50, lr=1e-3, seed=1),
    lambda: ifmm.ifmm_inv_check([np.eye(n) for n in (20, 100, 300, 700, 1100)]),
    lambda: [ifmm.ifmm_qr_check(np.eye(m, n), p, pivoted=q) for p in ("fp64", "fp32") for q in (False, True)
             for m, n in ((100, 10), (500, 200), (1500, 100), (900, 250), (4000, 90), (5000, 12))],
    lambda: [ifmm.ifmm_gemm_check(p, np.zeros((200, 100)), np.zeros((100, 200)))
             for p in ("fp64", "fp32", "bf16")],
    lambda: [svd(p, n) for p in (0, 1) for n in (10, 40, 100, 200, 300)],
    lambda: [top(n) for n in (30, 600, 2000)],
    lambda: [factor(p) for p in ("fp64", "fp32", "bf16")],
]
for dev in (0, 1, 0):
    fake.fake_set_device(dev)
    fake.fake_clear()
    for i, f in enumerate(calls):
        try:
            f()
        except ifmm.IFMMError as e:
            print("device", dev, "call", i, e)
    assert not refused(), refused()
"""


def test_every_launch_is_accepted_on_both_devices(tmp_path):
    kc = kernel_calls.compile_to(str(tmp_path / "libkernel_calls.so"))
    out = fake_runtime.run(SCRIPT.format(kc=kc), tmp_path)
    assert out == "", out
