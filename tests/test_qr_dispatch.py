"""Which kernels a QR block goes to, read from the launches of the host code: a tall
block of 17 to 64 columns is reduced by chunks of 256 rows while the stacked R
factors fit (1,536 rows), by larger chunks where they would not, and only then
goes to the one-CTA kernels in global memory; and the same with a lowered per-CTA
limit."""

import pytest

import fake_runtime

SCRIPT = r"""
def kernels(m, n, prec, piv):
    fake.fake_clear()
    ifmm.ifmm_qr_check(np.zeros((m, n)), prec, pivoted=piv)
    assert not refused()
    return launches("k_qr_reg"), launches("4k_qrI") + launches("6k_qrcpI")
for prec in ("fp32", "fp64"):
    for piv in (False, True):
        # the chunks (a short last one may be of another class) and the stacked block
        for m, n in {shapes}:
            reg, glob = kernels(m, n, prec, piv)
            assert reg in (2, 3) and glob == 0, (m, n, prec, piv, reg, glob)
        for m, n in {single}:
            assert kernels(m, n, prec, piv) == (1, 0), (m, n, prec, piv)
        # beyond 1536 rows of stacked factors of 1,536-row chunks
        assert kernels(37000, 64, prec, piv) == (0, 1)
"""
# 6,144 = 24 chunks of 256 rows; one more needs 512-row chunks, 12,289 needs 1,024, 24,577 needs 1,536
SHAPES = [(385, 17), (1000, 64), (6144, 64), (6145, 64), (6200, 64), (7000, 64), (8000, 60), (10000, 40), (12096, 64),
          (12289, 64), (24576, 64), (24577, 64), (36864, 64), (4000, 90)]
SINGLE = [(100, 16), (384, 64), (640, 130), (1536, 10), (500, 200)]


def test_tall_blocks_stay_in_registers(tmp_path):
    fake_runtime.run(SCRIPT.format(shapes=SHAPES, single=SINGLE), tmp_path)


LOWERED = r"""
fake.fake_clear()
for m, n in [(600, 20), (3000, 40), (200, 100), (60, 12)]:
    ifmm.ifmm_qr_check(np.zeros((m, n)), "fp64", pivoted=True)
assert not refused()
"""


@pytest.mark.parametrize("kb", [4, 24])
def test_lowered_limit(tmp_path, kb):
    fake_runtime.run(LOWERED, tmp_path, {"IFMM_QR_CTA_LIMIT_KB": str(kb)})
