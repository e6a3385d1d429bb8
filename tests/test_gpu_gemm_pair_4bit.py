"""The tests of the GEMMs on pairs of CTAs again without the kernel for few tokens, which takes most of their 4-bit products otherwise."""
import pytest

from tests import test_gpu_gemm_pair as pair
from tests.test_gpu_gemm_pair import (  # noqa: F401  (collected here too, under the fixture below)
    test_few_features_over_many_tokens_go_to_the_pairs, test_few_tiles_go_to_the_single_cta_kernel, test_gemm_chains_are_no_longer_than_the_single_cta_kernels,
    test_gemm_chains_of_products_that_both_kernels_take_as_fast, test_gemm_edges_match_oracle, test_gemm_with_the_least_workspace_keeps_the_chains_short,
    test_residual_in_a_tile_of_several_contributors, test_split_tiles_match_oracle_in_every_run_of_tokens, test_the_workspace_chooses_between_two_plans_only,
    test_tiles_of_several_contributors_match_oracle)

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def without_the_kernel_for_few_tokens(request, monkeypatch):
    from paper_2607_10183_b200 import binding as B
    if request.node.originalname != "test_split_tiles_that_no_flag_sends_to_the_pairs":
        context = B.Context
        monkeypatch.setattr(B, "Context", lambda *args, flags=0, **kw: context(*args, flags=flags | B.ATS_FLAG_NO_GEMM_FEW, **kw))


# Products with split tiles that run on the pairs as they are: two and more contributors, many tokens and few.
@pytest.mark.parametrize("fmt,N,K,T", [("q4", 10341, 12256, 135), ("q4", 5376, 8192, 986), ("mxfp4", 11776, 8960, 342)])
def test_split_tiles_that_no_flag_sends_to_the_pairs(fmt, N, K, T):
    pair.test_tiles_of_several_contributors_match_oracle(fmt, N, K, T)
