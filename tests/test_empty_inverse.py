"""Matrices of order 0 in a batch of inverses: nothing is launched for them (the
kernel's steps and its cluster barriers need a column) and their status is 0."""

import kernel_calls
import fake_runtime

SCRIPT = r"""
kc = ctypes.CDLL({kc!r})
def call(n):
    fake.fake_clear()
    A = np.zeros(sum(k * k for k in n) + 1)
    info = np.full(len(n), 7, np.int32)
    rc = kc.kc_inv(len(n), np.asarray(n, np.int32).ctypes.data_as(ctypes.c_void_p),
                   A.ctypes.data_as(ctypes.c_void_p), info.ctypes.data_as(ctypes.c_void_p))
    assert rc == 0, ifmm.lib.ifmm_last_error()
    return launches(""), info.tolist()
assert call([0, 0]) == (0, [0, 0])
k, info = call([0, 5, 0])
assert k == 1 and info[0] == info[2] == 0
"""


def test_order_zero(tmp_path):
    kc = kernel_calls.compile_to(str(tmp_path / "libkernel_calls.so"))
    fake_runtime.run(SCRIPT.format(kc=kc), tmp_path)
