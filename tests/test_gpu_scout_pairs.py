"""The short-video kernel (two CTAs a video) against the fp64 oracle at the
edges of its tiles and paths: frame counts around 4, 32, 64 and 128 (the
longest it takes), odd widths, and the widths where the row stride changes and
where a video leaves the kernel."""
import pytest
import torch

from paper_2608_24063_gb300 import synth
from paper_2608_24063_gb300 import viscache as vc
from test_gpu_scout import check_video

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("F,D", [(1, 1), (3, 5), (4, 33), (5, 31), (9, 700), (31, 64), (32, 512), (33, 130), (57, 100),
                                 (64, 710), (64, 711), (64, 751), (64, 752), (65, 300), (96, 97), (127, 288),
                                 (128, 288), (128, 290), (128, 297), (129, 64)])
def test_short_video_matches_oracle(F, D):
    H, t = synth.scout_embeddings(F * 11 + D, F, D)
    order, keys, gains, _ = vc.viscache_scout_mmr(H.to(DEV), t[None].to(DEV), [F], 0.7, (1, 1))
    torch.cuda.synchronize()
    assert check_video(H, t, 0.7, (1, 1), order, keys, gains.cpu()) <= 2
