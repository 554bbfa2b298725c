"""The CNN's stem rearrangement and max pool at odd image sizes, and the
classifiers at the edges of their image and class tiles, through whole forwards
against the fp64 oracle."""
import dataclasses

import numpy as np
import pytest

from helpers import dev, stream_handle
from oracle import resnet as orr
from oracle import vit as ov
from paper_2609_10018_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def _forward(model, img, classes):
    import torch
    x = dev(img)
    logits = torch.full((len(img), classes), float("nan"), dtype=torch.float32, device="cuda")
    model.forward(stream_handle(), x.data_ptr(), len(img), logits.data_ptr())
    model.sync_status(stream_handle())
    return logits.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("img,batch,classes,dtype", [
    (33, 17, 45, synth.BF16),   # odd image: single-value reads; 17 images, 45 classes: ragged classifier tiles
    (35, 3, 10, synth.F32),     # fp32 images
    (46, 33, 1000, synth.BF16),  # even image, odd pooled size
])
def test_resnet_odd_sizes(img, batch, classes, dtype):
    cfg = dataclasses.replace(synth.RESNET50, img=img, classes=classes, dtype=dtype)
    w, tables = synth.make_resnet_weights(cfg), synth.make_resnet_tables(cfg)
    x = synth.make_images(cfg, batch)
    pick = np.unique([0, 1, batch // 2, batch - 1])
    with binding.ElasticModel.resnet(cfg, w, tables[:1], max_batch=batch) as m:
        got = _forward(m, x, classes)
    assert np.all(np.isfinite(got))
    ref = orr.resnet_forward_sliced(ov.widen_all(w), cfg, tables[0]["a"], tables[0]["b"], x[pick])
    assert np.max(np.abs(got[pick] - ref)) <= 1e-2 * np.max(np.abs(ref))  # the library's parity bound


@pytest.mark.parametrize("batch,classes,dim,heads", [
    (15, 7, 192, 3),     # largest batch of the small classifier, fewer classes than warps
    (16, 33, 192, 3),    # smallest batch of the tiled one, one class past a tile
    (65, 45, 320, 5),    # one image past two tiles, d not a multiple of a chunk
    (1, 1000, 1024, 16),  # widest row
    (2, 600000, 64, 1),   # more groups of 8 classes than a grid has rows
])
def test_vit_classifier_tiles(batch, classes, dim, heads):
    cfg = synth.vit_small_variant(synth.TINY, dim=dim, heads=heads, mlp=64, layers=1, classes=classes,
                                  mode_heads=(heads,), mode_mlp=(64,))
    w, tables = synth.make_vit_weights(cfg), synth.make_vit_tables(cfg)
    x = synth.make_images(cfg, batch)
    with binding.ElasticModel.vit(cfg, w, tables, max_batch=batch) as m:
        got = _forward(m, x, classes)
    assert np.all(np.isfinite(got))
    ref = ov.vit_forward_sliced(ov.widen_all(w), cfg, tables[0]["heads"], tables[0]["mlp"], x)
    assert np.max(np.abs(got - ref)) <= 1e-2 * np.max(np.abs(ref))  # the library's parity bound
