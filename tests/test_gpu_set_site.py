"""ctm_set_site after graphs were captured: the kept graphs read the new tensor's packs."""
import pytest

from paper_2509_05090_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(precision="fp64"), dict(precision="split_bf16", n_split=5)])
@pytest.mark.parametrize("D,chi", [(2, 8), (4, 32), (6, 24)])
def test_steps_match_a_fresh_context(ctm_lib, D, chi, kw):
    """One-step, multi-step and ctm_converge's graphs from the same environment.  The arithmetic is a
    fresh context's but for the order of the QR's atomic sums: 1e-9 of the spectrum's norm, the bound
    of ctm_converge after ctm_set_site (test_gpu_paths.py)."""
    from paper_2509_05090_gb300 import binding
    A1, A2 = I.random_site_tensor(2, D, 11), I.random_site_tensor(2, D, 12)
    g = binding.CTM(A1, chi, **kw)
    f = binding.CTM(A2, chi, **kw)
    runs = [lambda x: x.ctm_step(1), lambda x: x.ctm_step(3),
            lambda x: x.ctm_converge(max_steps=4, tol=1e-30, check_every=2)]
    g.ctm_step(1)
    for run in runs:
        run(g)
    g.ctm_set_site(A2)
    f.ctm_step(4)
    for run in runs:
        g.ctm_set_env(*f.ctm_get_env())
        run(f)
        run(g)
        s, t = (x.ctm_get_intermediate("s") for x in (g, f))
        assert float((s - t).norm()) <= 1e-9 * float(t.norm())
    g.close()
    f.close()
