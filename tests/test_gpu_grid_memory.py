"""Device memory a grid keeps: in recurrence mode the checkpoints, the coefficients and the lists of tiles
and rings, not what only its set-up needs (the first degree above the polar cut at every order and ring,
20 MB on the grid below)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402


def test_recurrence_grid_keeps_no_setup_memory():
    nlat, nlon, lmax = 40000, 512, 255
    L, nh = lmax + 1, nlat // 2
    seg = sum((L - m + 15) // 16 for m in range(L))       # 16-degree segments of every order
    ckpt = 2 * seg * 2 * nh * 4                             # two parity planes, two FP32 values a node
    coef = L * 512 * 16
    tiles = 2 * L * ((nh + 127) // 128 + 1) * 16
    rings = nlat * (8 + 8 + 4 + 4 + 8) + nh * 8
    want = ckpt + coef + tiles + rings

    def grid():
        return shot.shot_grid_init(nlat, nlon, lmax, shot.SHOT_TF32X3, shot.SHOT_RECURRENCE)

    shot.shot_grid_free(grid())   # the kernels of the set-up are loaded
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    g = grid()
    try:
        kept = free0 - torch.cuda.mem_get_info()[0]
        assert want - 2 ** 20 <= kept <= want + 10 * 2 ** 20, (kept, want)   # allocations come in pages of 2 MB
    finally:
        shot.shot_grid_free(g)
