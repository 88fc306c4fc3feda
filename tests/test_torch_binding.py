"""The torch-tensor calls reject what they cannot marshal before anything reaches the library (no GPU needed)."""
import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def bd():
    from paper_2304_11267_b200 import binding
    from paper_2304_11267_b200 import build
    build.build()
    binding.load()
    return binding


@pytest.mark.parametrize("call", ["geglu", "groupnorm", "attention", "not a tensor", "argument count"])
def test_bad_tensors_raise(bd, call):
    x = torch.zeros(2, 4, 8, 8)
    if call == "geglu":
        with pytest.raises(ValueError):
            bd.geglu(x)
    elif call == "groupnorm":
        with pytest.raises(ValueError):
            bd.groupnorm(x, 2)
    elif call == "attention":
        with pytest.raises(ValueError):
            bd._ext().attention(None, bd.LAYOUT_BHND, x, x, x, None, None, None)
    elif call == "not a tensor":
        with pytest.raises(TypeError):
            bd.geglu([1.0, 2.0])
    else:
        with pytest.raises(TypeError):
            bd._ext().geglu(x)


@pytest.mark.skipif(torch.cuda.is_available(), reason="needs a machine whose CUDA calls fail")
def test_a_failing_device_is_an_error_and_not_an_answer(bd):
    """Which convolution is the faster one depends on the device; sizes that neither takes are answered without it."""
    assert not bd.sd_winograd_direct_preferred(1, 6, 127, 72, 40)
    with pytest.raises(bd.SdAttnError) as raised:
        bd.sd_winograd_direct_preferred(2, 64, 64, 320, 320)
    assert raised.value.status in (bd.ERR_CUDA, bd.ERR_ARCH)
