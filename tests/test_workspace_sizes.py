"""A workspace taken for the largest of several orders serves the others: the
size never shrinks with the order (no GPU needed)."""
import pytest


@pytest.fixture(scope="module")
def sk():
    from paper_1912_04062_gb300 import build
    build.build()
    import paper_1912_04062_gb300 as pkg
    pkg.lib()
    return pkg


# every order up to one past the first route limits, then around the later ones
ORDERS = list(range(2, 320)) + list(range(320, 17000, 97)) + [
    m + d for m in (3000, 3200, 4000, 4750, 8000, 11500, 16384) for d in (-1, 0, 1, 2)]


@pytest.mark.parametrize("vectors", [True, False])
@pytest.mark.parametrize("qtrd", ["SKEW_QTRD_AUTO", "SKEW_QTRD_FP32", "SKEW_QTRD_FP64", "SKEW_QTRD_DF"])
@pytest.mark.parametrize("mode", ["SKEW_MODE_FP64", "SKEW_MODE_MIXED_REFINED"])
@pytest.mark.parametrize("most", [10 ** 6, 1000, 33])
def test_size_never_shrinks_with_the_order(sk, mode, qtrd, vectors, most):
    opts = sk.Options(mode=getattr(sk, mode), qtrd=getattr(sk, qtrd))
    last = (0, None)
    for n in sorted(set(ORDERS)):
        size = sk.workspace_size(n, min(most, n // 2), opts, vectors=vectors)
        assert size >= last[0], (n, last)
        last = (size, n)
