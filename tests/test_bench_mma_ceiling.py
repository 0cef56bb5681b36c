"""The proposal's tensor ceiling in the bench line is one that its kernel cannot pass."""
import bench


def test_ceiling_is_above_what_the_kernel_does_and_below_the_dense_rate():
    cycles, tflops = bench.propose_mma_ceiling(512, 152)
    assert cycles == 6 * 50 + 25 * 80 + 25 * 64
    blocks = 2 ** 22 // 512
    flops = 2.0 * blocks * 512 * (9 * 32 + 2 * 9 * 32 * 32)
    # 2^22 bins take about 206 us with the median; the kernel alone cannot beat its own MMAs
    assert flops / 170e-6 / 1e12 < tflops
    assert tflops < 2.0 * 4096 * 152 * 2.07e9 / 1e12   # dense FP16: 4096 multiply-adds per SM and clock
    for hop in (256, 384):
        assert bench.propose_mma_ceiling(hop, 152)[1] < tflops
