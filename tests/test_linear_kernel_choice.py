"""Which kernel a linear takes, asked of the library on the CPU (148 SMs)."""
import pytest

from paper_2507_14959_b200 import binding

NONE, GELU, RESIDUAL, PATCH = 0, 1, 2, 3
TOKENS = 197


def test_arguments():
    for bad in ((100, 128, 1, NONE), (128, 100, 1, NONE), (128, 128, 0, NONE), (128, 128, 1, 4), (0, 128, 1, NONE)):
        with pytest.raises(binding.PolymorphError):
            binding.linear_kernel(*bad, adapters=False)
    with pytest.raises(binding.PolymorphError):
        binding.linear_kernel(128, 128, 1, NONE, False, n_sms=0)


@pytest.mark.parametrize("k_in,n_out,frames,width,split", [
    (3072, 768, 1, 64, 4), (3072, 768, 2, 128, 4), (3072, 768, 4, 128, 2), (3072, 768, 8, 192, 2), (3072, 768, 12, 256, 2), (3072, 768, 15, 256, 2),
    (2048, 512, 12, 256, 2), (2048, 512, 24, 256, 2), (4096, 1024, 6, 256, 2), (4096, 1024, 11, 256, 2), (3072, 768, 17, 192, 1)])
def test_long_k_with_adapters_is_split_while_the_sms_suffice(k_in, n_out, frames, width, split):
    """Each share of t keeps 16 significant bits there, which no other form does."""
    assert binding.linear_kernel(k_in, n_out, frames * TOKENS, RESIDUAL, True)[:3] == ("few rows", width, split)


@pytest.mark.parametrize("k_in,n_out,kernel", [(128, 640, "single"), (384, 896, "single"), (448, 1408, "single"), (576, 128, "single"), (640, 640, "pair"), (768, 640, "pair"), (3072, 128, "pair"),
                                               (384, 576, "pair"), (448, 1280, "pair"), (384, 1280, "single"), (384, 1152, "pair"), (768, 320, "single")])
@pytest.mark.parametrize("epilogue,adapters", [(NONE, True), (GELU, False), (RESIDUAL, True), (RESIDUAL, False)])
def test_widths_that_only_128_divides_take_pairs_for_long_k(k_in, n_out, kernel, epilogue, adapters):
    got = binding.linear_kernel(k_in, n_out, 300 * TOKENS, epilogue, adapters)
    assert got[0] == kernel
    if kernel == "pair" and n_out % 192 and n_out % 256:
        assert got[1] == 128


@pytest.mark.parametrize("k_in,n_out,frames,form", [
    (768, 768, 6, ("few rows", 64, 1)), (768, 768, 8, ("pair", 128, 1)), (768, 768, 14, ("pair", 128, 1)), (768, 768, 16, ("pair", 192, 1)),
    (1024, 1024, 10, ("pair", 128, 1)), (512, 512, 20, ("pair", 128, 1)), (512, 512, 24, ("few rows", 128, 1)), (512, 512, 28, ("pair", 256, 1)),
    (1280, 512, 24, ("few rows", 128, 1)), (2048, 512, 10, ("few rows", 128, 2)), (2048, 512, 12, ("pair", 128, 1)), (2048, 512, 24, ("few rows", 128, 1)),
    (256, 256, 20, ("few rows", 64, 1)), (256, 256, 40, ("few rows", 128, 1)), (256, 256, 96, ("single", 256, 1)), (384, 1024, 10, ("few rows", 128, 1)),
    (384, 384, 16, ("single", 128, 1)), (192, 192, 32, ("single", 128, 1)), (384, 768, 20, ("single", 256, 1)), (3072, 576, 4, ("few rows", 64, 2)),
    (3072, 576, 8, ("few rows", 64, 1)), (3072, 576, 12, ("few rows", 192, 2)), (3072, 576, 16, ("pair", 192, 1)), (3072, 768, 6, ("few rows", 128, 2)),
    (3072, 768, 8, ("pair", 128, 1)), (3072, 768, 12, ("pair", 128, 1)), (768, 320, 8, ("few rows", 64, 1))])
def test_residuals_without_adapters_leave_the_few_row_kernel_for_narrow_gemm_tiles_only(k_in, n_out, frames, form):
    assert binding.linear_kernel(k_in, n_out, frames * TOKENS, RESIDUAL, False)[:3] == form


@pytest.mark.parametrize("epilogue,threads", [(NONE, 576), (GELU, 576), (RESIDUAL, 576), (PATCH, 320)])
def test_epilogue_warps_of_256_wide_pair_tiles(epilogue, threads):
    """A warp per 64 columns of a lane quarter; patch placement, which stores by thread, keeps eight warps."""
    assert binding.linear_kernel(768, 768, 256 * 196, epilogue, epilogue != PATCH) == ("pair", 256, 1, threads)
