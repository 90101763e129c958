"""Prefill packs the prompts' rows into chunks of any requests: prompts that end
inside a row tile, span two chunks (more than 2304 rows in all), or hold a single
token, against the oracle (caches, draft caches, root, one step)."""
import pytest

from paper_2505_14260_gb300 import msd, synth
from tests.parity_support import run_parity

pytestmark = pytest.mark.gpu

TINY = synth.WORKLOADS["tiny"]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("batch,vis,text,requests", [
    (1, (0,), (1, 1), None),                # one row, no draft row
    (3, (0,), (1, 2), None),                # single-token prompts among others
    (4, (0, 64, 63), (1, 70), None),        # ends at, before and past row-tile edges
    (3, (2000, 2300), (20, 300), (1,)),     # three chunks: request 1 spans two
])
def test_packed_prefill_matches_oracle(dtype, batch, vis, text, requests):
    wl = TINY.with_(dtype=dtype, batch=batch, n_vis=vis, n_text=text, n_sys=4)
    run_parity(wl, 1, requests)


@pytest.mark.parametrize("strategy", sorted(msd.DRAFT_INPUTS))
def test_packed_prefill_draft_inputs(strategy):
    wl = TINY.with_(dtype="bf16", batch=3, n_vis=(30, 90), n_text=(3, 50), n_sys=4, draft_input=strategy)
    run_parity(wl, 1, None)
