"""The decode step where its selection and its split of a group's pages change:
candidate counts around the rank-counting limits (96 blocks of a CTA, 256 of a
group), blocks per score CTA around multiples of four, batches that give large
clusters down to single CTAs, more pages per CTA than stages.  Integer inputs: kept sets bit-exact."""
import pytest

from tests.test_gpu_decode import run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topk,blocks", [
    (4, 5), (4, 7), (4, 96), (4, 97), (48, 130), (4, 256), (4, 257), (4, 259), (64, 300), (32, 300),
    (32, 8 * 256), (32, 8 * 256 + 1), (32, 16 * 256), (32, 16 * 256 + 1), (64, 8 * 256), (64, 8 * 256 + 3), (33, 15 * 256 + 2),
])
def test_candidate_counts(topk, blocks):
    run_case(1, 4, 1, 128, 128, topk, [64 * blocks + 17], seed=blocks + topk, exact=True)


@pytest.mark.parametrize("B,Hq,Hkv,topk", [
    (1, 1, 1, 64), (1, 8, 1, 1), (10, 16, 8, 32), (20, 16, 8, 7), (58, 16, 8, 5), (64, 8, 8, 32),
])
def test_cluster_sizes(B, Hq, Hkv, topk):
    # 1 .. 512 groups: from 13 or more CTAs per cluster down to 1; a short sequence leaves CTAs without pages
    lens = [64 * topk + 130 if b % 3 else 1 + 7 * b for b in range(B)]
    run_case(B, Hq, Hkv, 128, 128, topk, lens, seed=B + topk, exact=True)
