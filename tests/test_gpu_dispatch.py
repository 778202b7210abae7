"""Which kernel, and how many CTAs of it, a call of a given size is: rules that only change the time, so that no comparison of
outputs notices when a range of sizes ends up on the slower side."""
import json
import re

import numpy as np
import pytest

import iodf_synth as S
from test_gpu_parity import G, _check_both_ways, _t  # noqa: F401  (G: the fixture)
from test_gpu_residual import _both_ways

pytestmark = pytest.mark.gpu


def _launches(fn, tmp_path):
    """(kernel name, CTAs, bytes of shared memory of a CTA) of what fn launches."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA], acc_events=True) as prof:
        fn()
        torch.cuda.synchronize()
    trace = tmp_path / "trace.json"
    prof.export_chrome_trace(str(trace))
    events = [e for e in json.loads(trace.read_text())["traceEvents"] if e.get("cat") == "kernel"]
    if not events:
        pytest.skip("kernel activity is not recorded here")
    return [(re.search(r"\w+_kernel", e["name"]).group(), int(np.prod(e["args"]["grid"])), e["args"]["shared memory"])
            for e in sorted(events, key=lambda e: e["ts"])]


@pytest.mark.parametrize("block,line", [(0, 24), (1, 12)])       # with prior parameters; the final block, of one scale
@pytest.mark.parametrize("more", [0, 1])
def test_streams_take_half_a_warp_above_a_line(G, block, line, more, tmp_path):
    import torch
    per_image = 16                                               # streams of an image to a block
    B = line * torch.cuda.get_device_properties(0).multi_processor_count // per_image + more
    model = S.make_model(0xFF00, 3, 32, 32, [True, False], 1, 16)
    d, d_fact = 3 * 32 * 32, 6 * 256
    m = G.iodf_create(model, B)
    codec = G.iodf_codec_create(m, S.logistic_codec(elems_per_stream=96))
    rng = np.random.default_rng(block)
    z = torch.from_numpy(rng.integers(-40, 41, (B, d)).astype(np.int32)).cuda()
    prior = torch.from_numpy(np.stack([rng.integers(-9, 10, (B, d_fact)), np.full((B, d_fact), 20)], axis=1).astype(np.int32)).cuda()
    words, counts = G.iodf_rans_encode(codec, z, prior)
    assert counts.shape == (B, 2 * per_image)
    out = torch.zeros_like(z)
    run = _launches(lambda: G.iodf_rans_decode_block(codec, block, words, counts, prior, out), tmp_path)
    G.iodf_codec_check(codec)
    part = slice(0, d_fact) if block == 0 else slice(d_fact, d)
    assert torch.equal(out[:, part], z[:, part])
    assert [name for name, _, _ in run] == ["rans_decode_half_kernel" if more else "rans_decode_kernel"]


@pytest.mark.parametrize("hidden,batch,plan,blocks", [
    (32, 2, 0, 1),           # convs of one chunk: the exchange of edges costs more than the halved multiply time
    (33, 2, 0, 2),           # two chunks
    (97, 2, 0, 2),           # four, the last ragged
    (97, 2, 1, 1),           # ... one block of two tiles, without neighbours
    (33, 149, 0, 1),         # more images than half the SMs
])
def test_blocks_of_a_16x16_residual_image(G, hidden, batch, plan, blocks, tmp_path):
    model = S.make_residual_model(0xFF20 + hidden, 3, 32, 32, [True], 2, hidden, 2, prune=(0.4, 0.7))
    x = np.random.default_rng(hidden).integers(0, 256, (batch, 3, 32, 32), dtype=np.uint8)
    m = _both_ways(G, model, x, plan=plan)[0] if batch < 9 else G.iodf_create(model, batch, plan=plan)
    (name, ctas, _), = _launches(lambda: G.iodf_forward(m, _t(x)), tmp_path)
    assert (name, ctas) == ("res_flow_kernel", batch * blocks)
    G.iodf_check(m)


@pytest.mark.parametrize("in_c,hidden,copies", [
    (2, 16, False),
    (16, 48, False),         # four units of the last conv, one for each of an image's four warps
    (18, 48, True),          # five
    (24, 130, True),
    (2, 512, True),          # streamed weights: the hidden layers' blocks are shared out
])
def test_copies_of_4x4_images_where_there_is_work_to_share(G, in_c, hidden, copies, tmp_path):
    """With copies one image's operands take as many rows as those of two or four, and a CTA's shared memory grows by the other images'
    flow variables alone."""
    model = S.make_model(0xFF40 + in_c + hidden, in_c, 8, 8, [True], 3, hidden)
    x = np.random.default_rng(in_c).integers(0, 256, (299, in_c, 8, 8), dtype=np.uint8)
    smem = []
    for batch in (1, 299):                                # the last CTA of 299 is not full
        m, _ = _check_both_ways(G, model, x[:batch], sample=None if batch == 1 else [0, 1, 297, 298])
        images = G.iodf_level_images_per_cta(m, 0)
        assert images == 1 if batch == 1 else images in (2, 4)
        (name, ctas, smem_cta), = _launches(lambda: G.iodf_forward(m, _t(x[:batch])), tmp_path)
        assert (name, ctas) == ("flow_level_kernel", (batch + images - 1) // images)
        smem.append(smem_cta)
    variables = (images - 1) * 4 * in_c * 16 * 4
    assert (smem[1] - smem[0] < variables + 128) == copies, smem
