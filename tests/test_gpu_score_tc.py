"""The tensor engine at the edges of its tiles: strips of 128 rows of W in pairs, chunks of 32 and distance products of 64
observations, features padded to 16 and split over stages of 64, one or two buffers of scaled candidates, and tiles whose pairs
of strips are shared out to several thread blocks.  Every element against the FP64 oracle (tolerances of ``tests/parity.py``).
"""
import numpy as np
import pytest

from paper_2604_11109_b200 import binding as b
from tests.test_gpu_parity import compare_everything, dev, fit_gpu, rand_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,n,d,m", [
    (1, 31, 4, 130),          # one chunk of a distance product is padding
    (1, 64, 16, 129),         # exactly one product; a tile of one candidate
    (1, 65, 17, 257),         # one observation in the second product
    (2, 128, 32, 300),        # exactly one strip; the FP32 copy of the candidates at its widest
    (1, 129, 33, 200),        # a second strip of 64 rows, without that copy
    (3, 192, 9, 140),         # a strip and a half, several GPs
    (1, 256, 64, 200),        # exactly one pair; one stage of features at its widest
    (2, 257, 65, 150),        # a pair and a strip of 64 rows; features split over two stages; pairs shared out
    (1, 385, 97, 260),        # two pairs; the second stage mostly padding
    (1, 641, 128, 300),       # an odd number of strips; one buffer of candidates
    (1, 1025, 21, 100),       # five pairs shared out
    (1, 1793, 40, 131),       # FP8 cross terms, eight pairs shared out
    (1, 300, 3, 200), (1, 300, 8, 200), (1, 300, 12, 200),   # one, two and four groups of four features in close pairs
    (1, 1800, 7, 140),                # the same with FP8 cross terms
    (1, 40, 5, 148 * 128 * 2 + 77),   # more tiles than thread blocks, ragged tail
    (1, 300, 12, 148 * 128 + 1),      # the same with two pairs
])
def test_edges_of_strips_chunks_stages_and_parts(batch, n, d, m):
    g = rand_problem(7000 + n + d, batch, n, d, m)
    gp = fit_gpu(g, b.ENGINE_TENSOR)
    assert b.r3_gp_engine(gp) == b.ENGINE_TENSOR
    compare_everything(g, gp, min(8, m), f"edges n{n} d{d} m{m}")
    gp.close()


def test_parts_of_a_tile_add_up_to_the_whole():
    """A pool of one tile, whose pairs of strips go to several thread blocks, and the same rows among enough others that every
    tile stays with one block: FP64 sums of the same FP32 parts in another order, so at most a last bit apart.  A smooth, noisy
    response, of which nothing is recomputed: what the FP64 pass has rewritten would not show the engine's sums."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = rand_problem(91, 1, 900, 24, sms * 128 * 16, sn2=0.1)
    g["Xcand"] = np.clip(g["Xcand"], 0, 1)
    g["y"] = (0.2 * g["y"] + 2 * np.sin(3 * g["X"].sum(2) / np.sqrt(24))).astype(np.float32)
    gp = fit_gpu(g, b.ENGINE_TENSOR)
    whole = [t[0, :100].clone() for t in b.r3_gp_score(gp, dev(g["Xcand"]))]
    assert b.r3_gp_last_rescued(gp) == 0
    part = [t[0] for t in b.r3_gp_score(gp, dev(g["Xcand"][:, :100]))]
    assert b.r3_gp_last_rescued(gp) == 0
    for a, c in zip(part[:2], whole[:2]):
        ulp = torch.finfo(torch.float32).eps * c.abs().clamp_min(1e-30)
        assert ((a - c).abs() <= ulp).all()
    gp.close()


@pytest.mark.parametrize("batch,n,d,m", [
    (1, 1900, 20, (7 * 148 + 200) * 128 - 31),   # FP8 cross terms: the tiles that decide, and seven waves, then one
    (1, 1900, 70, (7 * 148 + 10) * 128),         # less than what the first piece takes
    (2, 1850, 12, (5 * 148 + 3) * 128 + 1),      # several GPs: whole ones
    (1, 700, 20, 16 * 148 * 128 - 500),          # FP16 cross terms, three pieces
])
def test_pieces_of_a_host_pool_give_what_the_whole_gives(batch, n, d, m):
    g = rand_problem(7900 + n + d, batch, n, d, m)
    gp = fit_gpu(g, b.ENGINE_TENSOR)
    k = 20
    want = [t.cpu() for t in b.r3_gp_score_topk(gp, dev(g["Xcand"]), k)]
    b.r3_gp_check(gp)
    out = [torch.empty(batch, m).pin_memory() for _ in range(3)]
    out += [torch.empty(batch, k, dtype=torch.int32).pin_memory(), torch.empty(batch, k).pin_memory()]
    b.r3_gp_score_topk_host(gp, torch.from_numpy(g["Xcand"]).pin_memory(), k, tuple(out))
    b.r3_gp_check(gp)
    for a, c in zip(out, want):
        assert torch.equal(a, c)
    gp.close()
