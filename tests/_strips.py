"""Lattices that step in skewed strips, and how they are cut on a device with
129 MiB of L2: (shape, pair, storage, strips along z, along y)."""
L2_BYTES = 129 << 20

PLANS = [
    ((128, 96, 80), "27x19", "fp32", 4, 1),     # strips along z
    ((640, 150, 17), "19x7", "fp32", 1, 4),     # along y
    ((160, 160, 160), "27x19", "fp32", 4, 4),   # both, a cube
    ((129, 161, 99), "27x27", "fp32", 2, 5),    # odd sides, flat launches, uneven cuts
    ((96, 34, 330), "19x7", "fp32", 3, 1),      # a long box
    ((1024, 96, 96), "27x19", "fp16", 3, 3),    # pairs of nodes
    ((171, 160, 150), "19x7", "bf16", 2, 1),    # one node per thread in 16 bits
]
# larger ones, whose order of steps is looked at without running them
LARGE = [
    ((256, 256, 256), "27x19", "fp32", 6, 6),
    ((512, 512, 512), "27x19", "fp32", 16, 16),
    ((256, 256, 256), "27x19", "fp16", 12, 1),
    ((401, 203, 111), "15x7", "fp32", 3, 5),
]
