"""Host arithmetic of the W4A16 kernels' schedules: no GPU needed."""
import pytest

from paper_2605_13915_b200 import binding

SM_SHARED, CTA_RESERVED = 228 * 1024, 1024        # shared memory of an SM, and what the system takes of it per CTA


@pytest.fixture(autouse=True)
def _options():
    yield
    binding.debug_reset_options()


@pytest.mark.parametrize("M", [1, 16, 33, 128])
@pytest.mark.parametrize("N,K", [(2048, 2048), (1000, 2176), (4096, 4096), (2048, 14336)])
def test_few_token_clusters_have_their_sms_to_themselves(M, N, K):
    """A CTA holds all tensor memory of its SM while it waits for the CTAs of its cluster, so two of them must not share an SM: each
    asks for more than half of the shared memory, whatever its pipeline needs."""
    seen = 0
    for kw in (1, 2, 4):
        for S in range(2, 9):
            for h in (96, 128):
                binding.debug_set_option("MSD_W4_DECODE", 100000 * kw + 1000 * S + h)
                kernel, rows, cluster, splits, smem = binding.debug_gemm_w4a16_schedule(M, N, K)
                if kernel != 2:
                    continue                      # (a shape that does not fit)
                assert (rows, cluster, splits) == (h, S, S)
                assert 2 * (smem + CTA_RESERVED) > SM_SHARED, (kw, S, h, smem)
                seen += 1
    assert seen


@pytest.mark.parametrize("tokens", [1, 16, 32, 64, 96, 128])
@pytest.mark.parametrize("groups", [1, 8, 23, 64])
def test_grouped_pipelines_have_two_stages(groups, tokens):
    """A CTA that goes through several stages, of one tile or of several, needs room for two: the next is loaded while one is multiplied."""
    for N, K in [(4096, 1024), (5632, 896), (2048, 512), (7168, 2048), (1000, 128), (2048, 7168)]:
        _, _, stages, steps, _ = binding.debug_grouped_gemm_w4a16_schedule([tokens] * groups, N, K)
        assert steps >= 1 and stages >= min(2, steps), (N, K, stages, steps)


@pytest.mark.parametrize("tokens,E,N,K,kernel", [(16, 32, 2048, 7168, 2), (128, 32, 2048, 7168, 0), (96, 64, 7168, 2048, 0), (128, 8, 7168, 2048, 0),
                                                 (128, 23, 4096, 1024, 0), (1, 64, 4096, 1024, 2), (64, 8, 2048, 7168, 2)])
def test_grouped_calls_with_long_groups_take_token_tiles(tokens, E, N, K, kernel):
    """Both sides of the line between bands of weight rows (few tokens) and token tiles; empty groups do not count."""
    assert binding.debug_grouped_gemm_w4a16_schedule([tokens] * E, N, K)[0] == kernel
    assert binding.debug_grouped_gemm_w4a16_schedule([0, tokens] * E, N, K)[0] == kernel
    binding.debug_set_option("MSD_W4_DECODE", 0)
    assert binding.debug_grouped_gemm_w4a16_schedule([tokens] * E, N, K)[0] == 0


@pytest.mark.parametrize("M,N,K,kernel", [(95, 19288, 7040, 0), (79, 19712, 2432, 0), (16, 19288, 7040, 2), (1, 4096, 14336, 2), (64, 14336, 4096, 2)])
def test_layers_take_the_shorter_kernel(M, N, K, kernel):
    """Both sides of the line between bands of weight rows and token tiles, on shapes whose K neither of them splits; the same when the
    choice is remembered."""
    for _ in range(2):
        assert binding.debug_gemm_w4a16_schedule(M, N, K)[0] == kernel
