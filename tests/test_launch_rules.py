"""Host-side checks of the rules that pick how a step is launched, compiled from the solver's
header."""
from tests.test_checkpoint_route import answers


def test_stage_ctas_do_not_pile_up_beside_the_finalisation(tmp_path):
    """The stage kernel starts early unless an FP64 batch of one wave, with room for more CTAs on an
    SM than its even share, meets a finalisation on a quarter of the SMs: CTAs, CTAs that fit an SM,
    finalisation blocks."""
    cases = [
        (120, 3, 120, False),   # ten half channels of 5 x 3 x 11 nodes, 45 cells, V = 4 at eight cells
        (240, 5, 120, False),   # the same at V = 1 and eight cells
        (480, 5, 120, True),    # and four cells: four CTAs of five on an SM, nothing to pile up
        (60, 2, 120, False),
        (80, 1, 120, True),     # one CTA fits
        (32, 4, 8, True),       # one small channel: every CTA finds an empty SM
        (128, 2, 32, True),     # one C2 channel at V = 1: the finalisation holds a fifth of the SMs
        (112, 3, 38, True),     # together no more than the SMs
        (115, 3, 38, False),
        (5632, 3, 256, True),   # many waves
    ]
    got = answers(tmp_path, "".join('std::printf("%%d %%d ", stage_starts_early(false, %d, %d, %d), '
                                    'stage_starts_early(true, %d, %d, %d));\n' % (c[:3] + c[:3]) for c in cases))
    assert [g == "1" for g in got] == [v for c in cases for v in (c[3], True)]


def test_long_tiles_are_not_finalised_inside_the_stage_kernel(tmp_path):
    """fuse = 1 folds the finalisation into the stage kernel for tiles of up to eight cells; one CTA
    would finalise a longer one four cells after four.  The other modes never fold it."""
    got = answers(tmp_path, """
    for (int fuse : {0, 1, 2})
        for (int ZT : {3, 4, 8, 9, 16, 64}) std::printf("%d ", fold_finalisation(fuse, ZT));""")
    assert [g == "1" for g in got] == [f == 1 and z <= 8 for f in (0, 1, 2) for z in (3, 4, 8, 9, 16, 64)]
