"""(M, N, K, symmetric) of more than 128 tokens by the arrangement that w4a8_linear takes for them on a B200 (148 SMs, 33
clusters of four CTAs of the pair kernel): what test_gpu_prefill_arrangements.py runs, and what test_prefill_plan.py holds
prefill_choice to, so that a change of the rule which takes an arrangement's shapes away from its tests does not pass."""
SMS, QUADS = 148, 33

# in the order of PrefillKind in csrc/w4a8_prefill_plan.h
KINDS = ["pairs256", "pairs512", "pairs_k_cut", "whole64", "whole128", "whole256", "cut128", "cut256"]

SHAPES = {
    "pairs256": [(512, 6144, 4096, True), (700, 12304, 2048, False)],
    "pairs512": [(1061, 16384, 1024, True), (1152, 7648, 2560, False)],
    "pairs_k_cut": [(511, 2048, 8192, True), (300, 2064, 8320, False)],
    # one k-block more than the ring holds, and fewer; ragged last tiles on both sides
    "whole64": [(129, 1040, 2944, True), (200, 4080, 4096, True), (144, 992, 128, False)],
    "whole128": [(241, 8592, 5248, True), (400, 2560, 1408, False), (966, 944, 128, True)],
    # a launch of 145 CTAs, several rounds, two k-blocks
    "whole256": [(1196, 3680, 4864, False), (6573, 1360, 1920, True), (819, 4640, 128, False)],
    # K cut between 8, 5 and 4 CTAs: evenly, 97 and 51 k-blocks unevenly; ragged last tiles, a last token tile of one token
    "cut128": [(250, 1008, 8192, True), (151, 1072, 12416, False), (145, 1968, 6528, True), (257, 640, 8192, False)],
    # between 4 to 7 CTAs, a last token tile of a few tokens
    "cut256": [(193, 4000, 14336, False), (668, 1104, 10240, False), (130, 2432, 9856, True)],
}
