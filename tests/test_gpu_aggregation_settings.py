"""Which aggregation settings a handle takes: 2 and 4 chunks per lane and the mixed
layout where D spans that many chunks of 8 (rounded up to a power of two) and the
costs are bytes.  What is refused leaves the setting as it was."""
import pytest

torch = pytest.importorskip("torch")
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cost", [sgm.SGM_COST_CENSUS, sgm.SGM_COST_SAD])
@pytest.mark.parametrize("D", [1, 8, 9, 16, 17, 31, 48, 64, 65, 97, 128, 129, 192, 255])
def test_settings_are_taken_where_d_spans_them(D, cost):
    chunks = 1
    while 8 * chunks < D:
        chunks *= 2
    p = sgm.SgmParams(census_w=5, census_h=5, path_mask=0xF, P1=20, P2=80, cost=cost)
    with sgm.Handle(40, 12, D, p) as h:
        sgm.sgm_set_aggregation(h, 3, 1)
        kept = (3, 1)
        for setting, needs in ((1, 1), (2, 2), (sgm.SGM_AGG_CHUNKS_MIXED, 2), (4, 4)):
            if needs == 1 or (needs <= chunks and cost == sgm.SGM_COST_CENSUS):
                sgm.sgm_set_aggregation(h, 4, setting)
                kept = (4, setting)
            else:
                with pytest.raises(sgm.SgmError) as e:
                    sgm.sgm_set_aggregation(h, 4, setting)
                assert e.value.status == sgm.SGM_ERR_UNSUPPORTED
            assert sgm.sgm_get_aggregation(h) == kept
