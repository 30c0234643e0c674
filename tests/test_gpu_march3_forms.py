"""The forms of the FP32 3D z-marches beside the one the dispatch takes: the 3D tests again with the
widest lanes everywhere and with the scalar form everywhere (MPDATA_MARCH3, read once per process).
And the dispatch's choice on fields of few planes or few rows, by time."""
import os
import subprocess
import sys

import pytest

from test_gpu_dispatch_times import problem3, times

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("form", ["0", "2"], ids=["scalar", "widest"])
def test_3d_tests_pass_with_one_form_everywhere(form):
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider",
                        os.path.join(HERE, "test_gpu_march3_cells.py"), os.path.join(HERE, "test_gpu_3d.py")],
                       env={**os.environ, "MPDATA_MARCH3": form}, cwd=os.path.dirname(HERE), capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-3000:]


@pytest.mark.parametrize("shape,part", [((4, 100, 100), (4, 100, 60)), ((4, 32, 200), (4, 32, 60)), ((40, 32, 100), (40, 32, 60))])
def test_a_field_on_few_blocks_takes_the_time_of_a_narrower_one(shape, part):
    """With most SMs idle, more columns of blocks cost nothing: a slower form for them would."""
    whole, narrow = times(problem3(shape), problem3(part))
    assert whole <= 1.2 * narrow, (whole, narrow)
