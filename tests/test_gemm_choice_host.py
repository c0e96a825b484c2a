"""Which kernel SmoothGEMM takes (xy_gemm_choice), for the device the time models were fitted on: 148 SMs,
clusters of 1 .. 8 CTAs and of 1 .. 4 pairs as the occupancy query counts them there."""
import pytest

from paper_2412_18106_b200 import gemm as xg

B200 = [148, 148, 74, 45, 33, 26, 22, 15, 15, 74, 33, 22, 15]
SCRATCH = 2 * 148 * 128 * 256 * 4


# Shapes whose cut for the weight-major kernel (with scratch) has this many MMAs per K step and this many pairs that
# share K: every form the kernel has, in one, two and several token tiles, ragged in M, N and K.
FORMS = [(130, 12296, 520, 1, 1), (257, 6152, 1096, 1, 1), (200, 264, 328, 1, 1), (130, 6152, 3080, 1, 2), (257, 3080, 3080, 1, 2),
         (513, 2056, 3080, 1, 2), (130, 4104, 2056, 1, 3), (257, 2056, 2056, 1, 3), (200, 776, 2056, 1, 3), (130, 3080, 2056, 1, 4),
         (200, 1544, 3080, 1, 4), (130, 264, 2056, 1, 4), (257, 18696, 2056, 2, 1), (518, 6152, 6152, 2, 1), (1500, 3080, 1032, 2, 1),
         (257, 6152, 8200, 2, 2), (573, 3080, 8200, 2, 2), (781, 2056, 8200, 2, 2), (257, 4104, 6152, 2, 3), (1028, 1544, 6152, 2, 3),
         (257, 3080, 10248, 2, 4)]


def choice(M, N, K, scratch=SCRATCH, device=B200):
    return xg.xy_gemm_choice(M, N, K, scratch, device)


# Measured (us): what is chosen against the weight-major kernel.
@pytest.mark.parametrize("M,N,K,scratch,kernel,tile_n", [
    (352, 10240, 8192, 0, "tile", 256),        # 64 / 74
    (384, 10240, 8192, SCRATCH, "tile", 256),  # 64 / 73
    (448, 4096, 512, 0, "tile", 128),          # 6.8 / 8.5
    (512, 4096, 512, SCRATCH, "tile", 128),    # 6.8 / 8.8
    (1025, 4096, 512, 0, "tile", 256),         # 8.6 / 12.2
    (1500, 1032, 2304, 0, "tile", 128),        # 14 / 18
    (333, 256, 28672, SCRATCH, "split_k", 128),  # 22 / 30
    (1024, 8, 512, SCRATCH, "tile", 128),      # 5.3 / 8.6
    (820, 10240, 8192, 0, "tile", 256),        # 119 / 124
])
def test_kernels_that_beat_the_weight_major_one_are_taken(M, N, K, scratch, kernel, tile_n):
    c = choice(M, N, K, scratch)
    assert (c["kernel"], c["tile_n"]) == (kernel, tile_n), c


# Measured (us): the weight-major kernel against the one that would run otherwise.
@pytest.mark.parametrize("M,N,K,scratch", [
    (600, 28672, 4096, 0),              # 112 / 130
    (333, 28672, 4096, SCRATCH),        # 73 / 86
    (333, 4096, 14336, SCRATCH),        # 40 / 63
    (333, 6144, 4096, SCRATCH),         # 21 / 23
    (129, 57344, 8192, 0),              # 181 / 234
    (820, 3584, 18944, SCRATCH),        # 93 / 134
])
def test_the_weight_major_kernel_is_taken_where_it_is_faster(M, N, K, scratch):
    assert choice(M, N, K, scratch)["kernel"] == "weight_major"


def test_a_device_without_room_for_pairs_takes_the_other_kernels():
    c = choice(333, 28672, 4096, device=B200[:9] + [0, 0, 0, 0])
    assert c["kernel"] == "tile" and c["tok"] == 0
    assert choice(333, 28672, 4096, device=[1] + [1] + [0] * 7 + [0] * 4)["kernel"] == "tile"


@pytest.mark.parametrize("M", [1, 128, 129, 255, 333, 512, 513, 1025, 1536, 1537, 4096])
@pytest.mark.parametrize("N,K", [(8, 8), (4096, 14336), (131072, 8192), (1032, 2304)])
def test_cuts_cover_the_tokens_and_fit(M, N, K):
    for scratch in (0, SCRATCH):
        c = choice(M, N, K, scratch)
        if c["kernel"] != "weight_major":
            continue
        assert 128 < M <= 1536
        assert (c["m_tiles"] - 1) * c["tok"] < M <= c["m_tiles"] * c["tok"]
        assert c["tok"] % (16 * c["halves"]) == 0 and c["tok"] // c["halves"] <= 256 and c["halves"] in (1, 2)
        n_tiles = (N + 255) // 256
        if c["splits"] > 1:
            assert c["m_tiles"] * n_tiles * c["splits"] * c["tok"] * 1024 <= scratch
            assert c["m_tiles"] * n_tiles <= B200[8 + c["splits"]]


@pytest.mark.parametrize("scratch", [1024, SCRATCH // 2, SCRATCH - 16])
@pytest.mark.parametrize("M,N,K", [(200, 4096, 14336), (333, 4096, 14336), (200, 4096, 4096), (700, 2048, 4096)])
def test_too_little_scratch_is_none(M, N, K, scratch):
    assert choice(M, N, K, scratch) == choice(M, N, K, 0)


# Up to 128 tokens: what is chosen against the weight-streaming kernel (measured, us) ...
@pytest.mark.parametrize("M,N,K,kernel,tile_n", [
    (128, 16384, 1024, "tile", 128),     # 10.2 / 14.4
    (80, 16384, 1024, "tile", 128),      # 9.9 / 11.8
    (128, 12288, 4096, "tile", 128),     # 24.8 / 27.0
    (128, 4096, 512, "tile", 128),       # 6.6 / 7.5
    (128, 8, 512, "tile", 128),          # 5.2 / 6.9
    (128, 256, 28672, "split_k", 128),   # 21.3 / 24.8
])
def test_kernels_that_beat_the_weight_streaming_one_are_taken(M, N, K, kernel, tile_n):
    c = choice(M, N, K)
    assert (c["kernel"], c["tile_n"]) == (kernel, tile_n), c


# ... and where that one is faster, with slices of K whose clusters run at once.
@pytest.mark.parametrize("M,N,K,splits", [
    (16, 12288, 4096, (2,)),        # 20.1; three slices 24.7
    (16, 6144, 4096, (4, 5)),
    (16, 28672, 4096, (1,)),        # 39.8; two 40.7
    (16, 4096, 14336, (7, 8)),      # 20.6; six 22.1
    (1, 4096, 512, (1,)),
    (64, 4096, 4096, (6, 8)),
])
def test_the_weight_streaming_kernel_is_cut_to_what_fits(M, N, K, splits):
    c = choice(M, N, K)
    assert c["kernel"] == "weight_streaming" and c["splits"] in splits, c


@pytest.mark.parametrize("device", [B200, [132, 132, 66, 42, 32, 25, 20, 16, 14, 66, 32, 20, 14],
                                    [148] + [148] + [0] * 7 + [0] * 4])
@pytest.mark.parametrize("M", [1, 17, 64, 128])
def test_no_slice_of_k_is_empty(M, device):
    for N in (8, 128, 4096, 12288, 40000, 131072):
        for K in list(range(8, 4200, 88)) + [14336, 28672]:
            c = choice(M, N, K, device=device)
            if c["kernel"] == "weight_streaming":
                chunks = (K + 63) // 64
                assert 1 <= c["splits"] <= 8 and device[c["splits"]] > 0
                assert (c["splits"] - 1) * -(-chunks // c["splits"]) < chunks


@pytest.mark.parametrize("M,N,K,halves,splits", FORMS)
def test_every_form_of_the_weight_major_kernel_has_a_shape(M, N, K, halves, splits):
    c = choice(M, N, K)
    assert (c["kernel"], c["halves"], c["splits"]) == ("weight_major", halves, splits), c


def test_shapes_of_the_gpu_tests_reach_what_they_name():
    """Without scratch, tests/test_gpu_gemm.py names the cluster split of K and single-CTA and pair tiles."""
    reached = [choice(M, N, K, 0)["kernel"] for M in (1, 16, 33, 100, 128, 129, 300, 512)
               for N, K in ((512, 4096), (4096, 1024), (1032, 2304), (4096, 14336))]
    assert reached.count("split_k") >= 4 and reached.count("weight_streaming") >= 12
    assert choice(1024, 4096, 512, 0)["kernel"] == "pair"
    c = choice(520, 28672, 128, 0)
    assert (c["kernel"], c["tile_n"]) == ("tile", 256)
