"""Workspace sizes of the forward through the radial layer (host side)."""
import paper_2609_35099_b200 as e3j

HIDDEN = 64


def _sizes(plan, n_nodes, n_edges):
    """(preferred, least) of the call on harmonics and of the call on edge vectors."""
    return [(full(plan, n_nodes, n_edges, HIDDEN), least(plan, n_nodes, n_edges, HIDDEN)) for full, least in (
        (e3j.e3j_conv_radial_fwd_workspace_bytes, e3j.e3j_conv_radial_fwd_least_workspace_bytes),
        (e3j.e3j_conv_radial_vec_fwd_workspace_bytes, e3j.e3j_conv_radial_vec_fwd_least_workspace_bytes))]


def test_the_least_workspace_has_no_room_for_the_weights():
    plan = e3j.e3j_plan_create("128x0e+128x1o", 3, None, 3)
    row = 4 * plan.n_paths * plan.n_channels
    limit = (2 << 30) // row                       # the longest list whose weights the preferred form writes
    for n_edges in (1000, 160_900, limit):
        for full, least in _sizes(plan, 3000, n_edges):
            assert full >= n_edges * row and least < full - n_edges * row // 2
    for full, least in _sizes(plan, 3000, limit + 1):
        assert full == least < row * limit


def test_a_workspace_for_a_long_list_serves_every_shorter_one():
    plan = e3j.e3j_plan_create("128x0e+128x1o", 3, None, 3)
    longest = [full for full, _ in _sizes(plan, 3000, 400_000)]
    for n_edges in (0, 1, 1000, 160_900, 322_638, 399_999):
        assert all(least <= have for (_, least), have in zip(_sizes(plan, 3000, n_edges), longest))


def test_plans_without_the_kernel_need_the_whole_workspace():
    for plan in (e3j.e3j_plan_create("8x0e+8x1o", 2), e3j.e3j_plan_create("128x0e+128x1o", 3, None, 3, e3j.E3J_PLAN_RADIAL_MATERIALISE)):
        assert all(full == least for full, least in _sizes(plan, 100, 5000))
