"""n_tested counts every unordered candidate pair once: where each particle's
kernel reaches all others, it is n (n - 1) / 2, the number of in-range pairs,
and more kernels that reach less only lower both."""
import pytest

from paper_2506_06269_gb300 import ics
from gpu_helpers import gpu_step

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_06269_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n", [2, 17, 32, 33, 65, 100])
def test_pairs_tested_once(n, precision):
    b = ics.batch([ics.uniform_box(n, 3), ics.hernquist(3000, 4)])
    alone = ics.batch([ics.uniform_box(n, 3)])
    st = gpu_step(alone, [n - 1], [(0, 1e-3, 1.0)], [0.01], 1, 0, precision=precision)["stats"]
    assert st.n_pairs == n * (n - 1) // 2 and st.n_tested == n * (n - 1) // 2
    st = gpu_step(b, [n - 1, 32], [(0, 1e-3, 1.0)] * 2, [0.01] * 2, 1, 0, precision=precision)["stats"]
    assert st.n_pairs <= st.n_tested < (n * (n - 1) + 3000 * 2999) // 2
