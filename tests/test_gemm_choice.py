"""Which kernel a prompt product runs on, from the library's host logic: the products that the GPU tests mean for a kernel do reach it."""
import pytest

from tests import test_gpu_gemm_few as few
from tests import test_gpu_gemm_pair as pair
from tests import test_gpu_gemm_pair_4bit as pair_4bit


def _binding():
    from paper_2607_10183_b200 import build
    build.build()
    from paper_2607_10183_b200 import binding
    return binding


def _sets(test):
    """The parameter sets of a test, as dicts."""
    sets = [{}]
    for mark in test.pytestmark:
        if mark.name == "parametrize":
            names = [n.strip() for n in mark.args[0].split(",")]
            sets = [{**s, **dict(zip(names, v if len(names) > 1 else (v,)))} for s in sets for v in mark.args[1]]
    return sets


def _kernel(B, p, flags=0, fmt=None):
    fmt = {"q4": B.ATS_FMT_Q4B32, "mxfp4": B.ATS_FMT_MXFP4, "w16": B.ATS_FMT_W16}[fmt or p.get("fmt", "q4")]
    return B.host_gemm_kernel(fmt, p["N"], p["K"], p["T"], flags, 8 * p["T"] * p["N"] * 4)[0]


def test_products_of_few_tokens_run_on_their_kernel():
    B = _binding()
    for p in _sets(few.test_gemm_of_few_tokens_matches_oracle):
        assert _kernel(B, p) == B.ATS_GEMM_FEW, p
        assert _kernel(B, p, B.ATS_FLAG_NO_GEMM_FEW) != B.ATS_GEMM_FEW, p


def test_tiles_of_several_contributors_run_on_the_pairs():
    B = _binding()
    for t in (pair.test_tiles_of_several_contributors_match_oracle, pair.test_few_features_over_many_tokens_go_to_the_pairs):
        for p in _sets(t):
            assert _kernel(B, p, B.ATS_FLAG_NO_GEMM_FEW) == B.ATS_GEMM_PAIRS, p
    for p in _sets(pair.test_few_tiles_go_to_the_single_cta_kernel):
        assert _kernel(B, p, B.ATS_FLAG_NO_GEMM_FEW) == (B.ATS_GEMM_PAIRS if p["pairs"] else B.ATS_GEMM_PLAIN), p
    for p in _sets(pair_4bit.test_split_tiles_that_no_flag_sends_to_the_pairs):
        assert _kernel(B, p) == B.ATS_GEMM_PAIRS, p


def test_flags_and_sizes():
    B = _binding()
    for T in (9, 77, 512, 2048, 4000):
        for fmt in (B.ATS_FMT_Q4B32, B.ATS_FMT_MXFP4, B.ATS_FMT_W16):
            for n, k in ((4096, 4096), (300, 288), (14336, 4096)):
                assert B.host_gemm_kernel(fmt, n, k, T, B.ATS_FLAG_NO_GEMM_PAIR)[0] != B.ATS_GEMM_PAIRS
                kernel, chain = B.host_gemm_kernel(fmt, n, k, T, B.ATS_FLAG_NO_GEMM_PAIR | B.ATS_FLAG_NO_GEMM_FEW)
                assert kernel == B.ATS_GEMM_PLAIN and 0 < chain <= (k + 63) // 64 * 64
                assert fmt != B.ATS_FMT_W16 or B.host_gemm_kernel(fmt, n, k, T)[0] != B.ATS_GEMM_FEW
    for bad in ((4096, 4096, 8), (4096, 4100, 9), (0, 4096, 9)):
        with pytest.raises(B.AtsError):
            B.host_gemm_kernel(B.ATS_FMT_Q4B32, *bad)
    with pytest.raises(B.AtsError):
        B.host_gemm_kernel(B.ATS_FMT_F16, 4096, 4096, 9)


def test_without_pairs_the_kernel_for_few_tokens_is_compared_with_plain_tiles():
    """Its chains are no longer than theirs (a unit of 256 k at least), and it takes what it is faster at than they are."""
    import random
    B = _binding()
    rng = random.Random(3)
    taken = 0
    for _ in range(3000):
        n, k, T = int(2 ** rng.uniform(0, 14.8)), 32 * int(2 ** rng.uniform(0, 9)), int(2 ** rng.uniform(3.3, 12))
        fmt = rng.choice([B.ATS_FMT_Q4B32, B.ATS_FMT_MXFP4])
        kernel, chain = B.host_gemm_kernel(fmt, n, k, T, B.ATS_FLAG_NO_GEMM_PAIR)
        if kernel == B.ATS_GEMM_FEW:
            taken += 1
            assert chain <= max(256, B.host_gemm_kernel(fmt, n, k, T, B.ATS_FLAG_NO_GEMM_PAIR | B.ATS_FLAG_NO_GEMM_FEW)[1]), (n, k, T)
    assert taken > 2000
    for fmt, n, k, T in ((B.ATS_FMT_Q4B32, 13392, 4896, 1391), (B.ATS_FMT_MXFP4, 5983, 13344, 114), (B.ATS_FMT_MXFP4, 11047, 11968, 174)):
        assert B.host_gemm_kernel(fmt, n, k, T, B.ATS_FLAG_NO_GEMM_PAIR)[0] == B.ATS_GEMM_FEW


def test_chains_of_few_tokens_are_no_longer_than_the_other_kernels():
    """With all the scratch that these want; with less, by no more than a quarter (see the kernel)."""
    import random
    B = _binding()
    rng = random.Random(5)
    taken = 0
    for _ in range(4000):
        n, k, T = int(2 ** rng.uniform(9, 14)), 32 * int(2 ** rng.uniform(4, 9)), int(2 ** rng.uniform(3.3, 12))
        fmt = rng.choice([B.ATS_FMT_Q4B32, B.ATS_FMT_MXFP4])
        for scratch, more in ((1 << 40, 1.0), (32 * n * T, 1.25)):
            kernel, chain = B.host_gemm_kernel(fmt, n, k, T, 0, scratch)
            if kernel == B.ATS_GEMM_FEW:
                taken += 1
                assert chain <= max(256, more * B.host_gemm_kernel(fmt, n, k, T, B.ATS_FLAG_NO_GEMM_FEW, scratch)[1]), (n, k, T, scratch)
    assert taken > 5000
