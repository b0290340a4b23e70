"""Grouped problems are packed as structs: the same bytes, or the same refusal, as a
ctypes constructor for each gives, whatever a caller hands over."""
import numpy as np
import pytest

from tests.test_abi import ks  # noqa: F401  (builds the library)

BASE = dict(M=3, N=4, K=5, transA="N", transB="T", alpha=1.0, beta=0.0, A=0x1000, lda=5, B=0x2000, ldb=6, C=0x3000,
            ldc=7)


class Index:
    def __index__(self):
        return 7


def constructed(ks, q):
    return bytes(ks.Problem(q["M"], q["N"], q["K"], ks._c(q["transA"]), ks._c(q["transB"]), q["alpha"], q["beta"],
                            ks.ptr(q["A"]), q["lda"], ks.ptr(q["B"]), q["ldb"], ks.ptr(q["C"]), q["ldc"]))


@pytest.mark.parametrize("change", [
    {}, dict(alpha=1e39), dict(beta=-1e300), dict(alpha=np.float64(3.5e38)), dict(alpha=float("inf")), dict(alpha=2),
    dict(alpha=np.float32(1.5)), dict(alpha=None), dict(alpha="1"), dict(alpha=10 ** 400), dict(M=-1), dict(M=2 ** 63),
    dict(M=np.int64(9)), dict(M=Index()), dict(M=3.0), dict(lda=-2 ** 63 - 1), dict(A=None), dict(A=-1), dict(C=2 ** 64),
    dict(transA="t"), dict(transA=b"N"), dict(transA=78), dict(transB=bytearray(b"N")), dict(transA=""),
    dict(transB="NT")], ids=lambda c: ",".join(c) or "plain")
def test_as_constructed(ks, change):  # noqa: F811
    q = {**BASE, **change}
    try:
        want = constructed(ks, q)
    except Exception as e:
        with pytest.raises(type(e)):
            ks._problems([BASE, q])
    else:
        assert bytes(ks._problems([BASE, q, BASE])) == constructed(ks, BASE) + want + constructed(ks, BASE)


def test_defaults(ks):  # noqa: F811
    q = {k: v for k, v in BASE.items() if k not in ("transA", "transB", "alpha", "beta")}
    assert bytes(ks._problems([q])) == constructed(ks, BASE)
