"""Bytes of the launch that makes frame A as float and the pyramid's levels: each frame
read once, in the input's format at level 0 and as floats above, and every float frame
written once.  A record's step says whether frame A is made, its radius the levels."""
import bench


def test_frames_launches_count_each_frame_once():
    def b(name, W, H, made_a, levels):
        return bench.kernel_bytes(dict(name=name, pairs=64, width=W, height=H, step=made_a, radius=levels, nx=0, ny=0), 2, 8)

    px = 1024 * 1024
    assert b("frames/L0", 1024, 1024, 1, 2) == 64 * (2 * px * 2 + px * 4 + 2 * (px // 4 + px // 16) * 4)
    assert b("frames/L0", 1024, 1024, 0, 2) == 64 * (2 * px * 2 + 2 * (px // 4 + px // 16) * 4)  # both frames warped
    assert b("frames/L0", 1024, 1024, 1, 0) == 64 * (px * 2 + px * 4)  # no pyramid: frame A alone
    assert b("frames/L2", 256, 256, 0, 1) == 64 * (2 * 256 * 256 * 4 + 2 * 128 * 128 * 4)
