"""Which form an FP64 cycle takes (smg_cycle_form, host only): at sizes where one form measured at least 1.25 times as fast
as the other, the faster one; it follows from the call's arguments alone; FP32 and BF16 cycles have one form."""
import pytest


@pytest.fixture(scope="module")
def smg():
    from paper_1212_6680_gb300 import build

    build.build()
    from paper_1212_6680_gb300 import smg as m

    return m


# (shape, cycle, vectors): microseconds an application on the plane kernels and in mode space, one GB300
MEASURED = [
    ((2048, 1, 1), (1, 0), 1, 14, 2350), ((300, 1, 1), (1, 1), 1, 9, 369), ((100, 1, 1), (1, 0), 1, 4, 152),
    ((8, 4, 1), (1, 1), 1, 16, 43), ((32, 1, 1024), (1, 0), 1, 220, 426), ((128, 64, 1), (1, 0), 1, 77, 153),
    ((2048, 64, 5), (1, 0), 1, 3098, 4483), ((512, 512, 512), (1, 0), 1, 64100, 137819),
    ((1280, 80, 80), (1, 0), 1, 11103, 20410), ((1024, 64, 64), (1, 0), 8, 17982, 62958),
    ((1280, 40, 24), (1, 1), 8, 16104, 26316), ((2048, 24, 16), (1, 0), 1, 3394, 4584),
    ((24, 20, 16), (1, 0), 1, 320, 82), ((128, 128, 128), (1, 0), 1, 2349, 971),
    ((128, 128, 128), (1, 1), 8, 14720, 8484), ((256, 256, 256), (1, 1), 1, 18893, 12473),
    ((384, 384, 384), (1, 1), 1, 86541, 56923), ((200, 200, 200), (1, 1), 1, 14086, 7441),
    ((1024, 64, 64), (1, 1), 1, 15536, 9054), ((768, 48, 48), (1, 0), 1, 4815, 2983),
    ((512, 32, 32), (1, 1), 8, 6880, 5324), ((512, 128, 96), (1, 1), 1, 12941, 7781),
    ((160, 80, 80), (1, 0), 1, 2138, 824), ((886, 11, 12), (1, 0), 1, 1434, 1117),
]


@pytest.mark.parametrize("shape,cycle,nb,planes,modes", MEASURED)
def test_the_faster_form_is_taken(smg, shape, cycle, nb, planes, modes):
    assert max(planes, modes) >= 1.25 * min(planes, modes)
    want = smg.SMG_FORM_PLANES if planes < modes else smg.SMG_FORM_MODES
    assert smg.smg_cycle_form(*shape, *cycle, "fp64", nb) == want


def test_fp32_and_bf16_cycles_run_in_mode_space(smg):
    for prec in ("fp32", "bf16"):
        for shape in ((1, 1, 1), (2048, 1, 1), (512, 512, 512)):
            assert smg.smg_cycle_form(*shape, 1, 0, prec, 1) == smg.SMG_FORM_MODES


@pytest.mark.parametrize("args", [(0, 4, 4, 1, 0, "fp64", 1), (2049, 4, 4, 1, 0, "fp64", 1), (4, 513, 4, 1, 0, "fp64", 1),
                                  (4, 4, 4097, 1, 0, "fp64", 1), (4, 4, 4, 0, 0, "fp64", 1), (4, 4, 4, 1, -1, "fp64", 1),
                                  (4, 4, 4, 1, 0, "fp64", 0), (4, 4, 4, 1, 0, "fp64", 65)])
def test_arguments_the_other_entry_points_refuse_are_refused(smg, args):
    with pytest.raises(smg.SMGError) as e:
        smg.smg_cycle_form(*args)
    assert e.value.code == smg.SMG_ERR_ARG


def test_every_size_has_a_form(smg):
    """The estimates stay in range at the ends of the sizes smg_setup takes."""
    for nx in (1, 2, 31, 32, 33, 160, 161, 256, 257, 512, 513, 1025, 1537, 2048):
        for ny in (1, 2, 33, 65, 129, 257, 512):
            for nz in (1, 2, 3, 255, 4096):
                for nb in (1, 64):
                    assert smg.smg_cycle_form(nx, ny, nz, 1, 1, "fp64", nb) in (0, 1)
