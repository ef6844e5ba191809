"""The planes a 3D system may have: up to 512 points, or exactly 1024 in FP32."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sub,dtype,ok", [((32, 16, 4), "f32", True), ((32, 16, 4), "f64", True),
                                          ((32, 32, 4), "f32", True), ((128, 8, 4), "f32", True),
                                          ((32, 32, 4), "f64", False), ((32, 17, 4), "f32", False),
                                          ((32, 24, 4), "f32", False), ((16, 63, 4), "f32", False),
                                          ((128, 5, 4), "f32", False), ((24, 32, 4), "f32", False),
                                          ((256, 4, 4), "f32", False)])
@pytest.mark.parametrize("nf", [3, 5])
def test_plane_limit(sub, dtype, ok, nf):
    import paper_1911_05769_gb300 as at
    n = tuple(2 * m for m in sub)
    if ok:
        at.System3D(n, sub, 2, [0.1] * nf, 1e-6, dtype=dtype).close()
        return
    with pytest.raises(at.AtError) as e:
        at.System3D(n, sub, 2, [0.1] * nf, 1e-6, dtype=dtype)
    assert e.value.code == at.AT_ERR_ARG
    assert "512" in at.at_last_error()
