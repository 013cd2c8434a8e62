"""How a refinement is launched (no GPU: the library runs on tests/fake_cudart.c):
one cooperative launch for a frame that fits on the chip, launches per round for a
larger one and where a cooperative launch does not fit the context, and no second
try after any other error."""

import pytest

from test_host_lifetimes import run  # noqa: F401  (the fixture)

CALL = """
def refine(H, W):
    h = handle()
    rc = lib.epic_refine(h, buf(0), buf(1), H, W, 3, buf(2), None, None)
    return rc, names(), [fake.fake_cooperative(i) for i in range(fake.fake_launches())]
def per_round(got):
    kinds = ["coeff" if "coeff_kernel" in n else "sor" if "sor_kernel" in n else "update" for n in got]
    return kinds == (["coeff"] + ["sor"] * 10 + ["update"]) * 5   # 60 half-sweeps, six a launch
"""


def test_one_cooperative_launch(run):  # noqa: F811
    run(CALL + """
rc, got, cooperative = refine(70, 90)
assert rc == 0 and len(got) == 1 and "sor_kernel" in got[0] and cooperative == [1], (rc, got, cooperative)
""")


def test_frames_of_several_waves(run):  # noqa: F811
    run(CALL + """
rc, got, cooperative = refine(800, 900)
assert rc == 0 and per_round(got) and not any(cooperative), (rc, got)
""")


def test_where_a_cooperative_launch_is_too_large(run):  # noqa: F811
    run(CALL + """
fake.fake_fail_cooperative(720)   # cudaErrorCooperativeLaunchTooLarge
rc, got, cooperative = refine(70, 90)
assert rc == 0 and per_round(got) and not any(cooperative), (rc, got)
""")


@pytest.mark.parametrize("error", [1, 701, 719])
def test_any_other_error_is_reported(run, error):  # noqa: F811
    run(CALL + f"""
fake.fake_fail_cooperative({error})
rc, got, _ = refine(70, 90)
assert rc == native.EPIC_ERR_CUDA and got == [], (rc, got)
""")
