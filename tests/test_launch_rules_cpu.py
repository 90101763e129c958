"""The launch rules of the tensor-core GEMMs, on the host: no two launches can hold
tensor memory that each other's CTAs wait for, and the accumulators' chains stay short."""
import ctypes
import itertools
import random

import pytest

SM_SMEM = 228 * 1024          # shared memory of an SM
RESERVED = 1024               # of it, per resident CTA, for the system
TMEM_COLS = 512               # tensor-memory columns of an SM


@pytest.fixture(scope="module")
def shape():
    from paper_2505_14260_gb300 import build, msd
    build.build()
    lib = msd.lib()

    def at(m, k, o, planes, glu=0, sms=152):
        out = msd.msd_gemm_shape()
        assert lib.msd_test_gemm_shape(m, k, o, planes, glu, sms, ctypes.byref(out)) == msd.MSD_OK
        return out
    return at


def _shapes():
    """Every token-row class of both kernels against narrow to wide outputs and short to
    long K, and random sizes between."""
    ms = list(range(1, 130)) + [144, 160, 176, 255, 257, 333, 500, 576, 700, 961, 1024, 1245, 1500, 2304, 5000]
    for m, k, o in itertools.product(ms, (8, 64, 256, 512, 1024, 4096, 11008), (1, 128, 320, 4096, 9472, 32000)):
        yield m, k, o
    rng = random.Random(5)
    for _ in range(3000):
        yield (int(2 ** rng.uniform(0, 12)), 8 * int(2 ** rng.uniform(0, 11)), int(2 ** rng.uniform(0, 15.5)))


def test_ctas_that_share_an_sm_fit_its_tensor_memory(shape):
    """A CTA keeps its columns while it waits for its cluster, and an allocation waits
    without a limit, so CTAs of any launches that fit an SM by their shared memory have
    to fit it by their columns. (Registers are left out: they may change with the
    compiler. The tree attention's CTAs: 97 KB and 256 columns, 193 KB and 512.)"""
    least = {256: 97 * 1024, 512: 193 * 1024}       # columns -> least shared memory that a CTA holding them takes
    for m, k, o in _shapes():
        for planes, glu in ((1, 0), (2, 0), (2, 1)):
            g = shape(m, k, o, planes, glu)
            assert g.tmem_cols in (256, TMEM_COLS) and g.smem_bytes <= 227 * 1024     # (free columns are never scattered)
            least[g.tmem_cols] = min(least.get(g.tmem_cols, SM_SMEM), g.smem_bytes)
    for n in range(2, 9):
        for cols in itertools.combinations_with_replacement(sorted(least), n):
            if sum(least[c] + RESERVED for c in cols) <= SM_SMEM:
                assert sum(cols) <= TMEM_COLS, (cols, least)


def test_accumulator_chains_are_short(shape):
    """One-plane products (msd_linear): no accumulator of the many-row kernel adds up more
    than 32 K-blocks, none of the few-row kernel more than 16, or past 64 rows a quarter
    of K (two accumulators, two K splits: the room that the partial slices have)."""
    for m, k, o in _shapes():
        g = shape(m, k, o, 1)
        quarter = -(-(-(-k // 64)) // 4)
        assert g.chain <= (16 if m <= 64 else max(16, quarter) if m <= 128 else 32), (m, k, o, g.chain)


def test_shape_hook_refuses_bad_arguments():
    from paper_2505_14260_gb300 import build, msd
    build.build()
    out = msd.msd_gemm_shape()
    for args in ((0, 8, 8, 1, 0, 152), (8, 0, 8, 1, 0, 152), (8, 8, 0, 1, 0, 152), (8, 8, 8, 3, 0, 152),
                 (8, 8, 8, 1, 1, 152), (8, 8, 8, 1, 0, 1)):
        assert msd.lib().msd_test_gemm_shape(*args, ctypes.byref(out)) == msd.MSD_ERR_INVALID
    assert msd.lib().msd_test_gemm_shape(8, 8, 8, 1, 0, 152, None) == msd.MSD_ERR_INVALID
