"""Workspace sizes (host arithmetic, no GPU): one workspace, sized for the largest cube,
serves every smaller one, whatever the form."""
import pytest


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_sizes_grow_with_pixels_bands_and_components(prec):
    import paper_2403_18321_gb300 as g
    lib = g.load(build_if_missing=True)
    bands = (2, 3, 31, 63, 64, 100, 127, 128, 188, 191, 192, 255, 256)
    pixels = (2, 255, 1000, 10_000, 81_920, 207_400, 4_194_304)
    size = {(n, b, k): lib.pca_workspace_size(n, b, k, 0, prec)
            for n in pixels for b in bands for k in (1, 2)}
    for k in (1, 2):
        for n in pixels:
            for a, b in zip(bands, bands[1:]):
                assert 0 < size[n, a, k] <= size[n, b, k], (n, a, b, k)
        if prec < 2:       # (MIX: every processor gets the same number of slots)
            for b in bands:
                for n, m in zip(pixels, pixels[1:]):
                    assert size[n, b, k] <= size[m, b, k], (n, m, b, k)


def test_p64_partials_take_no_more_than_one_slot_per_256_pixels():
    """Slots of P64 partial sums: one per 256 pixels, 320 at most, as in P32."""
    import paper_2403_18321_gb300 as g
    lib = g.load(build_if_missing=True)
    for n, b in ((10_000, 100), (10_000, 50), (2000, 32), (1_000_000, 63), (122_500, 188)):
        slots = min(320, -(-n // 256))
        p32, p64 = (lib.pca_workspace_size(n, b, 1, 0, p) for p in (1, 0))
        assert p64 - p32 <= slots * 4 * (b * (b + 1) // 2) + 256, (n, b)
