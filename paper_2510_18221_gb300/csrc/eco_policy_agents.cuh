// eco_policy_agents.cuh -- the agents of one warp of k_policy
// (eco_policy_kernel.cuh): its loop over the alive list, included in the
// kernel's body where `few` is a constant or a variable.  A statement list,
// not a header: no include guard.

  const int w0 = few ? warp * (int)gridDim.x + (int)blockIdx.x : (int)blockIdx.x * WARPS + warp;
  // At the start of the launch every warp gathers an observation with no
  // weights in flight: the first 4 KB of each warp's first agent's weights
  // are requested into L2 before that gather.
  if (lane == 0 && w0 < G_eff && w0 < n_alive)
    prefetch_l2(d.wq + (int64_t)d.alive_list[w0] * L.stride, (uint32_t)min((int64_t)4096, (int64_t)L.off_w2));
  // The next agent's slot is read one agent ahead, and its environment,
  // cell and facing while the current agent's head is computed, so a new
  // agent starts with its observation gather.  (A slot's facing is written
  // only by the warp that computes it, in its own iteration.)
  int i = w0 < G_eff ? w0 : n_alive;
  // one-hot vision under the simple rules: cells_list's short cut
  const bool ahead = R.vision == VISION_CHANNELS && R.rules == RULES_SIMPLE && k * k <= 32 * kCellsAhead;
  int slot_n = 0, env_n = 0, pos_n = 0, f_n = 0;
  if (i < n_alive) {
    slot_n = d.alive_list[i];
    env_n = d.env_of[slot_n];
    pos_n = d.pos[slot_n];
    f_n = d.facing[slot_n];
  }
  for (; i < n_alive; i += G_eff) {
    const int slot = slot_n, env = env_n, pos = pos_n, f = f_n;
    const bool more = i + G_eff < n_alive;
    if (more) slot_n = d.alive_list[i + G_eff];
    if (!SPARSE && few) {
#pragma unroll
      for (int q = 0; q < kAheadBatches; ++q)
        prefetch_batch<UNROLL>(reinterpret_cast<const uint4 *>(d.wq + (int64_t)slot * L.stride) + 32 * UNROLL * q, lane);
    }
    if (env != e_cur) {
      flush();
      e_cur = env;
    }
    int nb_cell = 0;
    uint32_t nb_flags = 0;
    [[maybe_unused]] short *idx = reinterpret_cast<short *>(ls + 16);
    [[maybe_unused]] int n_nz = 0;
    if (SPARSE && ahead) {
      CellsAhead ca;
      cells_load(d, R, slot, env, pos, f, lane, kdiv, ca);
      n_nz = cells_list(R, ca, f, xs, idx, lane);
      nb_cell = ca.nb_cell;
      nb_flags = ca.nb_flags;
    } else {
      gather_obs(d, L, R, slot, env, pos, f, xs, lane, kdiv, &nb_cell, &nb_flags);
      if constexpr (SPARSE) {
        __syncwarp();
        n_nz = list_nonzero(L.D, xs, idx, lane);
      }
    }
    __syncwarp();

    const uint8_t *blk = d.wq + (int64_t)slot * L.stride;
    const uint4 *wb = reinterpret_cast<const uint4 *>(blk);
    const float *bias = reinterpret_cast<const float *>(blk + L.off_bias);
    const float *scale = reinterpret_cast<const float *>(blk + L.off_scale);

    // -- input layer: act(sum over sensors of (W_s x_s + b_s)) -> hs
    if constexpr (SPARSE) {
      layer_in_major<PREC, H, UNROLL, true, false>(wb + L.off_w1 / 16, n_nz, xs, bias, L.ns, scale, hs,
                                                   lane, L.relu, idx);
    } else {
      // one-hot vision: the patch inputs are 0 or 1, exact in f16
      const int n_exact = R.vision == VISION_CHANNELS ? L.patch : 0;
      if (few)
        layer_in_major<PREC, H, UNROLL, false, true>(wb + L.off_w1 / 16, L.D, xs, bias, L.ns, scale, hs, lane,
                                                     L.relu, nullptr, n_exact);
      else
        layer_in_major<PREC, H, UNROLL, false, false>(wb + L.off_w1 / 16, L.D, xs, bias, L.ns, scale, hs, lane,
                                                      L.relu, nullptr, n_exact);
    }
    __syncwarp();
    // -- hidden layers: h = act(W_l h + b_l), alternating between hs and xs
    float *cur = hs, *nxt = xs;
    for (int l = 0; l < L.L; ++l) {
      layer_in_major<PREC, H, UNROLL, false, false>(wb + (L.off_w2 + l * H * H * L.es) / 16, H, cur,
                                                    bias + L.ns * H + l * H, 1, scale + H + l * H, nxt,
                                                    lane, L.relu, nullptr);
      __syncwarp();
      float *tmp = cur;
      cur = nxt;
      nxt = tmp;
    }

    if (more) {
      env_n = d.env_of[slot_n];
      pos_n = d.pos[slot_n];
      f_n = d.facing[slot_n];
    }
    // -- head: logits = (W_out h [+ b_out]) / exp(tau) (output-major rows of
    //    H / E units; the temperature only in the paper form)
    const uint4 *w3 = wb + L.off_w3 / 16;
    const int U3 = L.A * UPJ;
    const float *hb = bias + L.ns * H + L.L * H;  // head bias, then tau
    const float tmul = L.temp ? expf(-__ldg(hb + (L.out_bias ? L.A : 0))) : 1.0f;
    // the head's groups of 32 units, up to kHeadBatch of them requested
    // before the first one is reduced
    constexpr int kHeadBatch = 4;
    for (int base = 0; base < U3; base += 32 * kHeadBatch) {
      uint4 hv[kHeadBatch];
#pragma unroll
      for (int g = 0; g < kHeadBatch; ++g) {
        const int u = base + 32 * g + lane;
        hv[g] = u < U3 ? ldg_stream(w3 + u) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int g = 0; g < kHeadBatch; ++g)
        if (base + 32 * g < U3)
          head_group<PREC, H>(hv[g], base + 32 * g + lane, U3, cur, scale + H + L.L * H, hb, L.out_bias,
                              L.temp, tmul, ls, lane);
    }
    __syncwarp();

    sample_and_claim(d, R, L.A, slot, env, pos, f, ls, lane, t, greedy, apply_moves, nb_cell, nb_flags, cnt);
    __syncwarp();
  }
