"""Host threads in the library at once: matrices of very different sizes
drawn side by side, each thread on its own stream, stay what they are when drawn
alone (the launch settings of one call must not reach another's)."""
import threading

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ccs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_01256_gb300 import build, ccs
    build.build()
    return ccs


def test_threads_draw_matrices(ccs):
    import torch
    # groups of ~20,000 entries, and of ~1000 as long as the large ones are drawn
    sizes = [(400003, 1000, 7), (300007, 700, 7), (2003, 500, 7), (1009, 300, 7)]
    drawn = [ccs.make_expander(n, m, d, 91) for n, m, d in sizes]
    errors, large = [], [2]
    start = threading.Barrier(len(sizes))

    def work(q, n, m, d, want):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                out = [torch.empty_like(t) for t in want]
                ws = ccs.workspace(ccs.ccs_workspace_size(ccs.OP_MAKE_EXPANDER, n, m, d))
                start.wait(60)
                rounds = 0
                while rounds < 2000 if q < 2 else large[0] > 0:
                    ccs.ccs_make_expander(n, m, d, 91, *out, ws)
                    rounds += 1
                for got, ref in zip(out, want):
                    assert torch.equal(got, ref)
        except BaseException as e:  # noqa: BLE001 -- reported by the test's thread
            errors.append(e)
        finally:
            large[0] -= q < 2

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(q, *size, want))
               for q, (size, want) in enumerate(zip(sizes, drawn))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
