"""The launch-shape table takes back whatever the tuner may have put there (host only): row-block
shapes (variant 5) of every tunable complex128 state count, which syk_autotune_apply tries."""
import json

import pytest

from paper_2002_05725_gb300 import syk


@pytest.mark.parametrize("batch", [1, 2, 4, 8, 16])
def test_complex128_row_block_entries(batch):
    syk.load(build_if_missing=True)
    syk.syk_autotune_reset()
    entry = {"N": 30, "dtype": 2, "batch": batch, "ntb": 7, "cluster": 4, "variant": 5}
    try:
        syk.syk_autotune_import(json.dumps({"apply_tiles": [entry]}))
        got = json.loads(syk.syk_autotune_export())["apply_tiles"]
        assert len(got) == 1 and all(got[0][k] == v for k, v in entry.items()), got
    finally:
        syk.syk_autotune_reset()
