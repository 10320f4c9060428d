"""The 16-bit rate of the tensor pipe is measured by its own probe: above its TF32 rate (nominally twice it), and a
probe that is not there is refused."""
import pytest

pytestmark = pytest.mark.gpu


def test_16bit_rate(R):
    tf32, f16 = R.rfdd_peak_probe(0), R.rfdd_peak_probe(4)
    assert 1.3 * tf32 < f16 < 2.6 * tf32
    assert R.rfdd_peak_probe(3) > 0.0
    with pytest.raises(R.RfddError) as e:
        R.rfdd_peak_probe(5)
    assert e.value.code == R.RFDD_EINVAL
