"""The library's fixed scratch array (apsm_train_noalloc) holds as long a sequence as the largest chunks allow: a
chunk that is shortened for speed (64 antennas with entries that leave) never costs a sequence its place. No GPU."""
import pytest

from paper_2201_05024_gb300 import apsm, build

SCRATCH = 8 << 20  # APSM_NOALLOC_SCRATCH_BYTES


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return apsm.load_library()


@pytest.mark.parametrize("K,W,D,longest", [(4, 13, 120, 2508), (4, 17, 120, 2420), (4, 17, 300, 2420), (4, 20, 300, 2376),
                                           (4, 24, 300, 1749), (16, 10, 300, 2478), (16, 17, 120, 2420),
                                           (16, 17, 300, 2365), (16, 20, 300, 2322), (16, 24, 120, 1696)])
def test_every_sequence_of_the_largest_chunks_fits(K, W, D, longest):
    """longest: the longest sequence that fits with the largest chunks shared memory allows."""
    p = apsm.Params(M=64, K=K, window=W, dict_cap=D, sigma=0.5, mu=0.5, eps=0.01, w_L=0.5)
    assert all(apsm.train_workspace_bytes(p, P) <= SCRATCH for P in range(1, longest + 1))
