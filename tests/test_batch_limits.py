"""Batch sizes refused on the host, before any device work."""
import pytest

from paper_2510_08288_gb300 import inputs


def test_batch_of_more_sampler_tiles_than_32_bits_count():
    """1,024 instances of one scenario and 2^31 - 1 steps: 2^35 tiles, 100 TB."""
    from paper_2510_08288_gb300 import build as B
    B.build()
    from paper_2510_08288_gb300 import rrg as R
    cfg = R.rrg_config_default(max_candidates=2, search=R.SEARCH_KSECTION, precision=R.FP32_RECHECK)
    with pytest.raises(R.RrgError) as e:
        R.rrg_batch_create(inputs.fc3_params(), cfg, [1] * 1024, [2 ** 31 - 1] * 1024)
    assert e.value.code == R.RRG_ENOMEM and "GB of scenarios" in str(e.value)
