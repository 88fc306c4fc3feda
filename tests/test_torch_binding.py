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
