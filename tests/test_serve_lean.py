"""Admission of jobs that fit the budget only without the cells of their images (host logic; no GPU): such a job is
admitted lean instead of being refused, one that doesn't fit either way is still refused."""
import numpy as np
import pytest

from paper_2412_14671_gb300.serve import EngineBackend, Job, MusterServer


class Backend:
    lean = EngineBackend.lean

    def footprint(self, job):
        from paper_2412_14671_gb300 import footprint

        return footprint(job.images.shape[1:], job.images.shape[0], **job.params)


def _job():
    return Job(7, np.zeros((3, 16, 20, 24), np.float32), dict(n_levels=1, steps_per_level=[2], window=3))


def test_a_job_that_fits_without_cells_is_admitted_lean():
    be = Backend()
    job = _job()
    full, lean = be.footprint(job), be.footprint(be.lean(job))
    assert lean < full
    for budget, plain, need in ((full, None, full), (full - 1, 1, lean), (lean, 1, lean)):
        srv = MusterServer(be, hbm_budget=budget)
        srv.submit(job)
        (queued, n), = srv.queue
        assert queued.id == job.id and queued.params.get("plain_images") == plain and n == need
    assert "plain_images" not in job.params  # the caller's job is not changed
    with pytest.raises(ValueError):
        MusterServer(be, hbm_budget=lean - 1).submit(job)
