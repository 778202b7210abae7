"""The compact level kernels at the edges of their ranges: shapes of tiles, ragged groups, widths on either side
of a dispatch, channels that need each form of requantisation, and the entropy coder's symbol look-up over
every range of scales; against the CPU oracle, bit for bit."""
import numpy as np
import pytest

import iodf_synth as S
import oracle as O
from test_gpu_parity import G, _check_both_ways, _t  # noqa: F401  (G: the fixture)
from test_gpu_residual import _both_ways

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_c", [1, 2, 3])
def test_whole_images_of_few_channels(G, in_c):
    """32 x 32 images whole in a CTA: two, four and six input channels in a record's eight bytes."""
    model = S.make_model(0xFA00 + in_c, in_c, 64, 64, [True], 2, 24)
    rng = np.random.default_rng(in_c)
    x = rng.integers(0, 256, (2, in_c, 64, 64), dtype=np.uint8)
    m, _ = _check_both_ways(G, model, x, plan=1)
    assert G.iodf_level_kernel_name(m, 0) == "flow_level_kernel" and G.iodf_level_images_per_cta(m, 0) == 1


@pytest.mark.parametrize("splits,hidden,batch,sample", [
    ([False], 16, 3, None),               # six channels in eight columns; the narrowest layers
    ([True], 33, 150, [0, 147, 149]),     # more images than SMs: two to a CTA, one alone
    ([True], 256, 2, None),               # nine blocks: the second GEMM's operand has one more than the third's
    ([True, True, True], 129, 1, None),   # 24 channels, as many columns as there are
    ([True, True, True], 160, 700, [0, 1, 349, 698, 699]),      # several to a CTA, the last with fewer
])
@pytest.mark.parametrize("plan", [0, 1])
def test_last_conv_on_8x8_frames(G, splits, hidden, batch, sample, plan):
    hw = 8 << len(splits)
    model = S.make_model(0xF800 + hw + hidden, 3, hw, hw, splits, 3, hidden)
    x = S.smooth_field_images(0xF900 + hw, batch, hw, hw, 2.0)
    _check_both_ways(G, model, x, sample=sample, plan=plan)


@pytest.mark.parametrize("in_c,hidden,batch,plan,sample", [
    (1, 16, 2, 0, None),                  # two translated channels: three products of eight columns, N rounded up
    (10, 129, 2, 0, None),                # twenty: 72 columns of 80; five blocks, the last conv starts after four
    (20, 129, 1, 0, None),                # forty in 48
    (28, 160, 1, 0, None),                # 56: wider than the hidden layer's columns, the last conv waits for all blocks
    (12, 192, 2, 1, None),                # two images whose accumulators do not fit side by side
    (12, 130, 2, 1, None),                # ... that do
    (12, 192, 600, 0, [0, 3, 596, 599]),  # four and more to a CTA: an MMA per tap
])
def test_last_conv_by_rows_of_taps(G, in_c, hidden, batch, plan, sample):
    model = S.make_model(0xFC00 + in_c + hidden, in_c, 16, 16, [False], 3, hidden)
    x = np.random.default_rng(in_c).integers(0, 256, (batch, in_c, 16, 16), dtype=np.uint8)
    _check_both_ways(G, model, x, sample=sample, plan=plan)


@pytest.mark.parametrize("in_c,hidden,batch,plan,sample", [
    (2, 16, 1, 0, None),                  # one image in one of four lane quarters, a block for one of four warps
    (6, 256, 1, 0, None),                 # nine blocks
    (24, 176, 3, 0, None),                # 96 channels, copies: the first and the last matrix share a slot
    (12, 512, 2, 0, None),                # streamed weights: copies in all lane quarters
    (4, 33, 3, 1, None),                  # several images to a CTA
    (12, 130, 299, 0, [0, 1, 297, 298]),  # two to a CTA, the last alone, and quarters without an image
])
def test_copies_of_4x4_images(G, in_c, hidden, batch, plan, sample):
    model = S.make_model(0xFD00 + in_c + hidden, in_c, 8, 8, [True], 3, hidden)
    x = np.random.default_rng(in_c).integers(0, 256, (batch, in_c, 8, 8), dtype=np.uint8)
    _check_both_ways(G, model, x, sample=sample, plan=plan)


@pytest.mark.parametrize("hw,splits,hidden,batch", [
    (16, [True, True], 16, 5),           # the last level 4 x 4: four images and one
    (16, [True, True], 31, 3),           # 8 x 8 tiles of 64 rows, six and twelve channels in
    (32, [True, True, True], 33, 2),     # 16 x 16: two tiles
    (48, [True], 16, 2),                 # 24 x 24: nine 64-row tiles
    (32, [False, True], 256, 2),         # the widest that can be resident
    (64, [True], 200, 1),                # eight tiles whose accumulators do not fit side by side: streamed
    (64, [True, True], 48, 1),           # 32 x 32 in eight blocks of one tile, then 16 x 16
    (64, [True], 48, 20),                # ... in four of two tiles
    (64, [False], 40, 40),               # ... in two of four
    (48, [True], 300, 2),                # 24 x 24 in blocks of 64-row tiles, streamed weights
    (64, [True, True], 257, 1),          # the narrowest streamed weights, eight tiles
    (32, [True, True, True], 24, 300),   # more images than SMs: two images of two tiles, two and four of one
    (16, [True, True], 24, 1190),        # eight images per CTA, the last with six
    (16, [True, True], 512, 6),          # the widest; 4 x 4 level with two ragged groups
])
@pytest.mark.parametrize("plan", [0, 1])
def test_three_conv_levels(G, hw, splits, hidden, batch, plan):
    model = S.make_model(0xF100 + hw + hidden, 3, hw, hw, splits, 3, hidden)
    x = S.smooth_field_images(0xF200 + hw, batch, hw, hw, 2.0)
    m, z = _check_both_ways(G, model, x, plan=plan)
    few, _ = G.iodf_forward(m, _t(x[-3:]))            # (the launch shape depends on the batch of the call)
    np.testing.assert_array_equal(few.cpu().numpy(), z[-3:])
    assert {G.iodf_level_kernel_name(m, k) for k in range(len(splits))} == {"flow_level_kernel"}


@pytest.mark.parametrize("hw,hidden,batch", [
    (64, 16, 1),         # 32 x 32 in eight blocks, every one with corners
    (64, 16, 20),        # ... in four
    (64, 272, 3),        # ... in eight, streamed weights
    (32, 16, 9),         # 16 x 16 in two blocks; fewer input words than threads per pixel pair
])
def test_split_images_through_long_chains(G, hw, hidden, batch):
    """Blocks of an image exchange edges and add to one another's accumulators at every coupling; short couplings, as
    many as a level can have, and the same call again and again: a sum that is added to before it has been cleared, or
    an edge that comes early, changes the latents."""
    import torch
    model = S.make_model(0xF600 + hw + hidden, 3, hw, hw, [True], 32 if hidden < 100 else 4, hidden)
    x = S.smooth_field_images(0xF700 + hw, batch, hw, hw, 2.0)
    m, z = _check_both_ways(G, model, x)
    xt, zt = _t(x), _t(z)
    for _ in range(20):
        assert torch.equal(G.iodf_forward(m, xt)[0], zt) and torch.equal(G.iodf_inverse(m, zt), xt)
    G.iodf_check(m)


@pytest.mark.parametrize("hidden,batch,images", [
    (96, 300, 1),        # three waves of one image 72 us, two of two images 80
    (96, 512, 2),        # four 96, two 82
    (256, 256, 2),       # two images, streamed weights 116 us; one image in two blocks, resident 127
    (288, 160, 2),       # streamed: two waves of one image in two blocks 119 us, one of two images 116
    (320, 200, 2),       # ... 125 and 120
])
def test_images_per_cta_follow_the_hidden_width(G, hidden, batch, images):
    """A 16 x 16 level of 24 channels: what a tile costs beside a coupling's serial part decides between more waves
    and more images per CTA."""
    m = G.iodf_create(S.make_model(0xFA00, 3, 64, 64, [True, True], 4, hidden), batch)
    assert G.iodf_level_images_per_cta(m, 1) == images


@pytest.mark.parametrize("hidden,images", [
    (256, [1, 1, 1, 4]),     # 8 x 8: two images' weights would be streamed, 41 us of an SM each against 35 for one
    (144, [1, 1, 2, 4]),     # everything resident: as many as a tile holds
    (512, [1, 1, 2, 4]),     # everything streamed: the same
])
def test_throughput_plan_takes_the_least_sm_time_per_image(G, hidden, images):
    model = S.make_model(0xFB00 + hidden, 3, 64, 64, [True] * 4, 4, hidden)
    x = S.smooth_field_images(0xFB01, 5, 64, 64, 2.0)
    m, _ = _check_both_ways(G, model, x, plan=G.IODF_PLAN_THROUGHPUT)
    assert [G.iodf_level_images_per_cta(m, k) for k in range(4)] == images


@pytest.mark.parametrize("hw,splits,couplings,hidden,blocks,prune,batch,plan", [
    (64, [True], 1, 128, 1, None, 1, 0),           # 32 x 32 in eight 8 x 16 blocks
    (64, [True], 1, 128, 1, None, 1, 1),           # ... in four 16 x 16 ones
    (32, [True], 2, 97, 2, (0.4, 0.7), 2, 0),      # 16 x 16: two blocks, four chunks with a ragged last one
    (16, [True], 1, 32, 1, None, 3, 0),            # 8 x 8: one chunk
    (8, [True], 1, 65, 2, None, 5, 1),             # 4 x 4: three images and two
])
def test_residual_levels(G, hw, splits, couplings, hidden, blocks, prune, batch, plan):
    model = S.make_residual_model(0xF300 + hw + hidden, 3, hw, hw, splits, couplings, hidden, blocks, prune=prune)
    x = S.smooth_field_images(0xF400 + hw, batch, hw, hw, 2.0)
    m, _, _ = _both_ways(G, model, x, plan=plan)
    assert {G.iodf_level_kernel_name(m, k) for k in range(len(splits))} == {"res_flow_kernel"}


@pytest.mark.parametrize("hidden,batch,plan", [(16, 1, 0), (16, 3, 1), (128, 2, 0)])
def test_residual_blocks_through_long_chains(G, hidden, batch, plan):
    """Blocks of an image send their edges after every conv, one conv ahead at most: the same call again and again."""
    import torch
    model = S.make_residual_model(0xF800 + hidden, 3, 64, 64, [True], 6 if hidden < 100 else 1, hidden, 4)
    x = S.smooth_field_images(0xF900, batch, 64, 64, 2.0)
    m, z, _ = _both_ways(G, model, x, plan=plan)
    xt, zt = _t(x), _t(z)
    for _ in range(20):
        assert torch.equal(G.iodf_forward(m, xt)[0], zt) and torch.equal(G.iodf_inverse(m, zt), xt)
    G.iodf_check(m)


@pytest.mark.parametrize("in_c,hw,hidden,prune,batch", [
    (6, 32, 128, (0.6, 0.9), 2),     # 16 x 16 in two blocks, 24 channels: three slots, convs of one, three and four chunks
    (3, 16, 96, None, 3),            # 8 x 8: four slots, three chunks everywhere
    (12, 8, 128, (0.4, 0.7), 2),     # 4 x 4: two to four chunks
])
def test_weight_slots_pass_between_the_warps_that_read_them(G, in_c, hw, hidden, prune, batch):
    """Levels of one tile have two warps that take a conv's chunks in turn, and with it a slot of the weight ring is now one's, now
    the other's: the same call again and again."""
    import torch
    model = S.make_residual_model(0xFE00 + hw, in_c, hw, hw, [True], 2, hidden, 4, prune=prune)
    x = np.random.default_rng(hw).integers(0, 256, (batch, in_c, hw, hw), dtype=np.uint8)
    m, z, _ = _both_ways(G, model, x)
    assert G.iodf_level_kernel_name(m, 0) == "res_flow_kernel"
    xt, zt = _t(x), _t(z)
    for _ in range(50):
        assert torch.equal(G.iodf_forward(m, xt)[0], zt) and torch.equal(G.iodf_inverse(m, zt), xt)
    G.iodf_check(m)


@pytest.mark.parametrize("per_sm,elems", [(0, 97), (24, 103), (25, 103), (40, 31), (41, 33)])   # streams per SM: up to 24 a warp each
@pytest.mark.parametrize("ls", [0, 20, 40, 63])                                                 # (one scale: 12), then half of one
def test_symbol_look_up_at_every_kind_of_scale(G, ls, per_sm, elems):
    """Residuals over the whole window at one scale: slots that mean one symbol and slots that mean hundreds."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = max(3, per_sm * sms // 15)                                             # 15 streams of an image to a block
    model = S.make_model(0xF500, 3, 32, 32, [True, False], 1, 16)
    codec = S.logistic_codec(elems_per_stream=elems)
    d, d_fact = 3 * 32 * 32, 6 * 256
    rng = np.random.default_rng(ls)
    prior = np.stack([rng.integers(-50, 50, (B, d_fact)), np.full((B, d_fact), ls)], axis=1).astype(np.int32)
    z = rng.integers(-2200, 2201, (B, d)).astype(np.int32)
    z[:, ::3] = rng.integers(-3, 4, z[:, ::3].shape)
    w_ref, c_ref = O.rans_encode(codec, model, z, prior)
    m = G.iodf_create(model, B)
    cd = G.iodf_codec_create(m, codec)
    words, counts = G.iodf_rans_encode(cd, _t(z), _t(prior))
    cc = counts.cpu().numpy().view(np.uint32)
    np.testing.assert_array_equal(cc, c_ref)
    w = words.cpu().numpy().view(np.uint16)
    valid = np.arange(w.shape[2])[None, None, :] < cc[:, :, None]
    np.testing.assert_array_equal(np.where(valid, w, 0), np.where(valid, w_ref, 0))
    out = torch.zeros((B, d), dtype=torch.int32, device="cuda")
    for q in range(cd.n_blocks):
        G.iodf_rans_decode_block(cd, q, words, counts, _t(prior), out)
    G.iodf_codec_check(cd)
    np.testing.assert_array_equal(out.cpu().numpy(), z)
    counts[B - 1, 0] -= 1                             # a stream that lacks its last word is noticed, the others are not touched
    out.zero_()
    G.iodf_rans_decode_block(cd, 0, words, counts, _t(prior), out)
    with pytest.raises(G.IodfError):
        G.iodf_codec_check(cd)
    np.testing.assert_array_equal(out.cpu().numpy()[:B - 1, :d_fact], z[:B - 1, :d_fact])


@pytest.mark.parametrize("umax,scales,elems", [
    (8192, 64, 1), (8192, 64, 7), (8192, 64, 8), (8192, 64, 9), (8192, 64, 300),
    (8192, 1024, 9),                      # the largest tables that a codec may have
    (5947, 64, 9), (5948, 64, 9), (6079, 64, 9), (6080, 64, 9),      # about 48 KB of shared memory
])
def test_coder_with_large_tables(G, umax, scales, elems):
    """The widest sigmoid tables, on either side of the shared memory that a kernel has without asking for it, and streams
    on either side of the encoder's batches of eight symbols, the last of a block shorter."""
    import torch
    model = S.make_model(0xF510, 3, 16, 16, [True], 1, 16)
    codec = S.logistic_codec(elems_per_stream=elems)
    codec["R"] = np.resize(codec["R"], scales)
    u = np.arange(-umax, umax + 1) / (umax / 16.0)
    codec.update(G=np.floor((65536 - 4097) / (1 + np.exp(-u)) + 0.5).astype(np.uint16), umax=umax)
    B, d, d_fact = 2, 3 * 16 * 16, 6 * 64
    rng = np.random.default_rng(elems)
    prior = np.stack([rng.integers(-50, 50, (B, d_fact)), rng.integers(0, 64, (B, d_fact))], axis=1).astype(np.int32)
    z = rng.integers(-2200, 2201, (B, d)).astype(np.int32)
    w_ref, c_ref = O.rans_encode(codec, model, z, prior)
    m = G.iodf_create(model, B)
    cd = G.iodf_codec_create(m, codec)
    words, counts = G.iodf_rans_encode(cd, _t(z), _t(prior))
    cc = counts.cpu().numpy().view(np.uint32)
    np.testing.assert_array_equal(cc, c_ref)
    w = words.cpu().numpy().view(np.uint16)
    valid = np.arange(w.shape[2])[None, None, :] < cc[:, :, None]
    np.testing.assert_array_equal(np.where(valid, w, 0), np.where(valid, w_ref, 0))
    out = torch.zeros((B, d), dtype=torch.int32, device="cuda")
    for q in range(cd.n_blocks):
        G.iodf_rans_decode_block(cd, q, words, counts, _t(prior), out)
    G.iodf_codec_check(cd)
    np.testing.assert_array_equal(out.cpu().numpy(), z)


_FIRST_CODEC = """
import sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
import iodf_synth as S
import paper_2206_08869_b200 as G
umax = int(sys.argv[2])
m = G.iodf_create(S.make_model(0xF520, 3, 16, 16, [True], 1, 16), 2)
codec = S.logistic_codec(umax=umax)
cd = G.iodf_codec_create(m, codec)
z, prior = G.iodf_forward(m, torch.from_numpy(S.smooth_field_images(0xF521, 2, 16, 16, 2.0)).cuda())
words, counts = G.iodf_rans_encode(cd, z, prior)
out = torch.zeros_like(z)
for q in range(cd.n_blocks):
    G.iodf_rans_decode_block(cd, q, words, counts, prior, out)
G.iodf_codec_check(cd)
print("equal", torch.equal(out, z))
"""


@pytest.mark.parametrize("umax", [
    5947,      # the encoder's dynamic and static shared memory together: 48 KB
    5948,      # ... 16 bytes more
    6079,      # its dynamic shared memory alone: 48 KB
    6080,      # ... 16 bytes more
])
def test_first_codec_of_a_process_about_48_kb(umax):
    """What shared memory a kernel may use is a state of the process, so each size is the first one of its own process."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _FIRST_CODEC, root, str(umax)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split()[-2:] == ["equal", "True"], r.stdout


def test_matrices_that_no_launch_shape_reads_are_not_kept(G):
    """Weights of an 8 x 8 level at width 512 are streamed, so that its last conv never runs in its direct form. 48 channels
    translated: that form's matrices would be 7 MB of 32 couplings' 32; the rest is the allocator's granularity."""
    import torch
    G.iodf_create(S.make_model(0xFC00, 3, 16, 16, [True], 1, 16), 1)          # (whatever is allocated only once)
    model = S.make_model(0xFC01, 24, 16, 16, [True], 32, 512)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    m = G.iodf_create(model, 1)
    taken = before - torch.cuda.mem_get_info()[0]
    assert G.iodf_level_kernel_name(m, 0) == "flow_level_kernel"
    first, second, last, meta = 512 * 36 * 16, 512 * 17 * 32, 432 * 16 * 32, 8192        # bytes of a coupling's parts
    prior = 96 * 36 * 16 + 8192
    assert taken <= 32 * (first + second + last + meta) + prior + (4 << 20)
