"""One batch of more frames than the association kernel stages at once, with
segments that split and join again: merges and better views change instances'
embeddings inside the batch, so gates taken at its start have to be taken
again; every counter and the final map equal the oracle's."""
import numpy as np
import pytest

import oracle
import synth
from tests import common

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_embeddings_changed_inside_a_long_batch(precision):
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    sc = synth.tiny_scene(num_frames=70)
    fr = sc.render(range(70))
    masks = sc.max_masks + 2
    cfg = common.disc_cfg(sc, max_masks=masks, batch_frames=128, precision=precision)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    gmap.set_schedule(batch_split=1)
    frames, counts = [], []
    for i in range(70):
        lab, n = fr.labels[i], int(fr.num_masks[i])
        if i % 4 != 0:  # the two largest masks cut in half
            for k in (1, 2):
                u = np.where((lab == k).any(axis=0))[0]
                half = lab[:, (u[0] + u[-1]) // 2:]
                half[half == k] = n + k
            n += 2
        counts.append(n)
        frames.append(device_frame(torch.from_numpy(fr.depth[i]).to(dev), torch.from_numpy(lab.view(np.int16)).to(dev),
                                   torch.from_numpy(fr.tokens[i]).to(dev), fr.poses[i], (sc.fx, sc.fy, sc.cx, sc.cy), n))
    stats, done, rc = gmap.integrate_frames(frames)
    assert rc == 0 and done == 70
    for i in range(70):
        o = omap.integrate(fr.depth[i], fr.labels[i], fr.tokens[i], fr.poses[i], (sc.fx, sc.fy, sc.cx, sc.cy), counts[i])
        for gk, ok in common.COUNT_FIELDS:
            assert stats[i][gk] == o[ok], f"frame {i} {gk}: {stats[i][gk]} vs {o[ok]}"
    common.compare_maps(gmap, omap, ctx="chain")
    assert sum(s["merges"] for s in stats) > 0
    assert sum(s["embedding_copies"] for s in stats) > sum(s["new_instances"] for s in stats)
    gmap.close()
