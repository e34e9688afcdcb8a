"""Sides no batch can hold are refused, whatever their size."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


@pytest.mark.parametrize("L", [2 ** 31 - 1, 2 ** 30 + 1, 46341, 1, 0, -5])
def test_refused(sw, L):
    for sides in ([L], [64, L]):
        with pytest.raises(sw.SWError) as ei:
            sw.sw_batch_create(sides, [0.4] * len(sides), [1] * len(sides))
        assert ei.value.status == sw.SW_EINVAL
