"""The measured ceiling that the transforms' rate is compared with runs the transforms' own butterfly."""
import pytest

pytestmark = pytest.mark.gpu


def test_butterfly_probe_multiplies_by_halves():
    """Cycles per butterfly and warp, an IMAD being two: the products by halves alone hold the multiply pipe for 26,
    a 64-bit Shoup butterfly holds it for 40.8, so a rate between the two is the former's."""
    import paper_2604_19890_gb300 as ssg
    cycles = 2 * ssg.alu_probe(0, 65536) / ssg.alu_probe(1, 16384)
    assert 26 < cycles < 40.8
