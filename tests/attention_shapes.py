"""Launch shapes of the attention tests and the kernel that each is there for.
tests/test_host_routes.py checks on the CPU that the cost rule takes it."""

# (layers, query heads, KV heads, page size, tokens per sequence, region-aligned),
# then the form of the first step's launch: (CTAs per item, warps, scores in
# scratch), or None where the pages depend on the regions
CLUSTER = [
    ((1, 8, 1, 16, [15], 0), (1, 4, False)),                          # one tile, one CTA
    ((1, 3, 1, 16, [431], 0), (8, 4, False)),                         # G = 3 padded heads
    ((1, 16, 2, 32, [1, 17, 4095], 0), (16, 8, False)),               # most chunks of the short ones are empty
    ((2, 28, 4, 32, [1000] * 3 + [33], 1), None),                     # half-empty second tiles
    ((1, 12, 2, 16, [1500 + 16 * i for i in range(12)], 0), (8, 4, False)),
    ((2, 16, 2, 16, [300 + 7 * i for i in range(40)], 0), (1, 4, False)),      # one CTA per item
    ((3, 5, 1, 16, [1790 - 25 * i for i in range(60)], 0), (1, 8, False)),     # the same, 8 warps, more than one wave
    ((1, 16, 2, 32, [20000, 17, 9001], 0), (16, 8, False)),           # 10 tiles per warp
    ((2, 8, 2, 16, [6100, 4000, 5999], 1), None),
    ((8, 7, 1, 16, [3500 + 50 * i for i in range(12)], 0), (1, 8, True)),      # 32 tiles per warp
]

# md_attend_mass_noalloc on the persistent kernel: (layers, query heads, KV
# heads, page size, tokens per sequence)
NOALLOC_PERSISTENT = [
    (1, 16, 2, 16, [20007 - 16 * i for i in range(8)]),     # 20 chunks per item and their partials
    (1, 8, 2, 32, [20017 - 32 * i for i in range(8)]),
    (15, 12, 2, 16, [1024 - (i % 3) for i in range(64)]),   # one chunk per item
    (15, 6, 2, 32, [1024 - (i % 3) for i in range(64)]),
]
