"""gdgs_project on its own writes its outputs and the projected splats, nothing for sorts
that do not follow."""
import pytest
import torch

import paper_2405_05446_gb300 as G
from paper_2405_05446_gb300 import scenes as S

from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu


def test_projection_alone_leaves_the_sorts_words():
    ensure_lib()
    sc, cam = S.tiny_scene(3, n=4, channels=3), S.tiny_camera(64, 48)
    g = G.gaussians_to_device(sc)
    ws = torch.full((G.workspace_size(sc.n, 3, 64, 48, None, None),), 0xAB, dtype=torch.uint8, device="cuda")
    G.project(g, cam, ws)
    assert G.sync_status(ws)["status"] == 0
    # the control block (below 4 KB, cleared) and at most 64 bytes a splat; the sorts' counts are 10 KB
    assert int((ws != 0xAB).sum()) <= 4096 + 64 * sc.n
