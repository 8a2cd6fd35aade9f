"""(M, N, K, symmetric) of up to 128 tokens by the kernel that w4a8_linear takes for them on a B200 (148 SMs, the clusters below
resident), given a workspace: on both sides of the limits of w4a8_decode_plan.h.  test_gpu_decode_kinds.py runs them, and
test_decode_plan.py holds decode_choice to them, so that a change of a rule which takes a kernel's shapes away from its tests does
not pass."""
SMS = 148
RESIDENT = [0, 148, 74, 45, 33, 26, 22, 15, 15]   # clusters of the persistent kernel, by CTAs in one

# in the order of DecodeKind in csrc/w4a8_decode_plan.h
KINDS = ["none", "direct", "whole", "cluster", "rows", "rows_half"]

SHAPES = {
    "direct": [
        (8, 1024, 1024, True), (1, 1024, 512, False),                    # at least 1024 channels
        (8, 4864, 640, True), (8, 3312, 640, False),                     # few tokens: 8000 K - 2 or 3 million weights
        (8, 4256, 2816, True), (7, 3536, 2816, False),                   # ... 12 or 10 million
        (4, 2048, 7168, True), (1, 4096, 4096, False), (3, 4736, 2304, False),   # one unit of work per warp
        (12, 2304, 1664, True), (9, 2048, 1408, False),                  # ... nine to twelve tokens
        (9, 2112, 1024, True), (16, 1232, 1792, False), (16, 3040, 2560, True),  # nine tokens and more
        (5, 1200, 640, False), (16, 2384, 1920, False)],                 # odd units per CTA, k-blocks that are no multiple of four
    "whole": [
        (8, 1008, 2304, True), (8, 4880, 640, True), (8, 3328, 640, False), (16, 2160, 1024, True), (13, 2304, 1664, True),
        (16, 4080, 2688, False), (16, 4080, 2944, True), (5, 4864, 2688, False),
        (8, 13184, 512, True), (16, 16000, 384, False),                  # more tiles than half the SMs
        (32, 18944, 1024, True), (33, 18944, 2432, True), (128, 18944, 3072, False), (65, 18944, 2304, True), (65, 18944, 2304, False),
        (17, 18960, 256, False), (124, 37904, 2048, True),               # more tiles than SMs
        (128, 9472, 2944, True), (17, 640, 1280, False),                 # few tiles, short K
        (120, 2048, 2944, False), (128, 7664, 5120, False)],             # few tiles, clusters do not pay
    "cluster": [(17, 640, 1408, False), (40, 8720, 2176, False), (32, 4096, 4096, True), (128, 4096, 14336, False), (65, 512, 8192, True)],
    "rows": [
        (5, 4128, 4480, True), (1, 4016, 5376, False), (1, 6144, 4096, True), (16, 3600, 3200, False), (13, 1024, 8320, True), (8, 2048, 8192, False), (5, 1120, 10624, False), (12, 1552, 14336, False),   # K cut
        (16, 128, 4096, True), (5, 16, 14336, False),
        (16, 28672, 1792, False), (3, 37904, 1792, True),                # one and two blocks of 128 rows, two runs a CTA
        (32, 18944, 1152, True), (33, 18944, 2560, True), (17, 18960, 384, False), (124, 37904, 2176, True),
        (128, 7664, 3072, True), (44, 6384, 1792, True),                 # few tiles, K not cut
        (128, 18944, 3200, False), (113, 18944, 4224, False)],           # as many stages as groups in both rings
    "rows_half": [
        (5, 4736, 3200, True), (4, 4128, 5120, False), (12, 2048, 6144, True), (8, 1008, 2432, True), (3, 1008, 6144, False),  # K cut
        (2, 16, 2560, True),
        (8, 13200, 512, True), (16, 16016, 384, False), (16, 18960, 256, True), (16, 28672, 1664, False), (3, 37904, 896, True)],
}
