// jx_rollout.cu — rollouts in two passes.
//
// The actions of a rollout are known in advance, so where every agent will
// stand after each step does not wait for any frame. The walk steps all
// agents, one lane per env, and leaves a camera record (24 bytes) per env and
// step. The draw renders every (env, step) frame from its record, in any
// order. Against one warp stepping and rendering an env through all its steps
// this
//  - takes the step logic off the warps that draw (it ran in all 32 lanes),
//  - leaves no chain of steps: a launch over few envs fills the chip, and
//  - lets blocks be handed out as they come: a warp's fixed share of envs
//    leaves the last SMs running alone, since the SMs' shares of a saturated
//    write path differ (pure frame writes: 6.3-6.6 TB/s in fixed shares, 7.6
//    TB/s in blocks handed out in order).
// The steps are cut into parts, and one launch walks a part while it draws the
// part before: the walk is a chain of short steps on few warps (about 1 us a
// step), the draw fills the memory system meanwhile. The blocks of the two
// share no data but through the launch before.
// An episode that ends within the rollout needs its env's next map: the walk
// stops that env before the step that ends the episode, the draw renders the
// frames up to there, and the env kernel, launched last, runs the env's
// remaining steps as in a launch of its own (generation included).
// The grayscale stack keeps an env's last four frames, so the draw writes only
// the planes of a part's last four.
#include "jx_device.cuh"
#include "jx_host.h"

namespace jx {
namespace {

constexpr int kActAhead = 8;  // steps of actions fetched ahead in the walk

// floor(v) for |v| < 2^21, offset by the bits of 1.5 * 2^23: one addition
// rounded down instead of two compares.
__device__ __forceinline__ int floor_bits(float v) { return __float_as_int(__fadd_rd(v, 12582912.f)); }
constexpr int kFloorZero = 0x4B400000;

// Which of the offsets -1, 0, 1 (bits 0, 1, 2) the interval [f - r, f + r]
// touches, f in [-1/2, 3/2] (floor_small of its ends and what lies between).
__device__ __forceinline__ uint32_t span3(float f, float r) {
  return (1u << (floor_bits(f + r) - (kFloorZero - 2))) - (1u << (floor_bits(f - r) - (kFloorZero - 1)));
}
// The rows of mask m (solid3x3) that `rows` selects, or-ed.
__device__ __forceinline__ uint32_t rows3(uint32_t m, uint32_t rows) {
  return ((rows & 1u) ? m : 0u) | ((rows & 2u) ? m >> 3 : 0u) | ((rows & 4u) ? m >> 6 : 0u);
}

__host__ __device__ __forceinline__ int walk_warp_bytes(int K) { return 32 * (4 * (K > 0 ? K : 1) + kActAhead); }

// One walk warp: 32 envs, a lane each, every lane through steps t_begin ..
// t_end - 1 of the rollout. Shared memory (walk_warp_bytes): the envs' event
// sprites and the actions ahead, word w (byte w) of lane l at [32 w + l], so
// that a lane reads only what it wrote and no two lanes share a bank.
// What bounds it is the length of a step's instruction chain on one warp: the
// cells around the agent are looked up only where it enters a cell, in a window
// of the env's bit plane that registers hold, the actions of 8 steps come with one round of loads, and the
// next step's turn-table entry is fetched a step ahead (turns depend on the
// actions alone).
// GRAY: as render_env's.
template <int GRAY>
__device__ __forceinline__ void walk_envs(const Params& p, int e, int t_begin, int t_end, uint32_t* sm, int lane) {
  const bool on = e < p.n;
  const int es = on ? e : p.n - 1;  // lanes past the last env load its state and store nothing
  const int S = p.S, sh = p.pitch_shift;
  uint32_t* const spr = sm;
  uint8_t* const acts = reinterpret_cast<uint8_t*>(spr + 32 * (p.K > 0 ? p.K : 1));
  const size_t stride = (size_t)p.out_stride;
  uint32_t ahead[kActAhead];
  const uint8_t* act = p.actions + (size_t)t_begin * stride + es;
#pragma unroll
  for (int i = 0; i < kActAhead; ++i) ahead[i] = t_begin + i < t_end ? act[i * stride] : 0u;
  Env r = load_env(p, es);
  // An earlier part may have stopped the env. A grayscale stack whose step count
  // comes from below zero (a state set by the host) is left to the env kernel:
  // the frame of step 0 writes all four planes, which no order of drawing keeps.
  int stop = t_begin == 0 ? (GRAY != 0 && p.gray && r.t < 0 ? 0 : p.steps) : p.stop[es];
  const int door_x = p.st.obj[6 * (size_t)es + 4], door_y = p.st.obj[6 * (size_t)es + 5];
  // the sprites that make events: cell x | cell y << 8 | type << 16
  int n_ev = 0;
  {
    const int nspr = p.st.nspr[es] > p.K ? p.K : p.st.nspr[es];
    for (int k = 0; k < nspr; ++k) {
      const size_t i = (size_t)es * p.K + k;
      const int type = p.st.spr_type[i];
      if (type != kSprGoal && key_colour(type) < 0) continue;
      const int x = (int)floorf(p.st.spr_x[i]), y = (int)floorf(p.st.spr_y[i]);
      if ((unsigned)x >= (unsigned)kMaxSide || (unsigned)y >= (unsigned)kMaxSide) continue;  // on no map
      spr[32 * n_ev++ + lane] = (uint32_t)(x | y << 8 | type << 16);
    }
  }
  const uint32_t* plane = plane_of(p, es);
  const uint8_t* map = p.st.map + (size_t)es * S * S;
  // An 8 x 8 window of the bit plane around the agent, in registers (bit
  // 8 dy + dx for cell (wx + dx, wy + dy), cells outside the map set): loads of
  // the map go out only when the agent nears its edge. Beside a draw that
  // saturates the memory system a load takes microseconds.
  uint32_t win_lo = 0u, win_hi = 0u;
  int wx = -64, wy = -64;
  auto load_window = [&]() {
    wx = r.cx - 3 < (1 << sh) - 8 ? r.cx - 3 : (1 << sh) - 8;
    wx = wx < 0 ? 0 : wx;
    wy = r.cy - 3 < S - 8 ? r.cy - 3 : S - 8;
    wy = wy < 0 ? 0 : wy;
    const int b = (wy << sh) + wx, w = 1 << (sh - 5);
    const uint32_t *q0 = plane + (b >> 5), *q1 = plane + ((b + 7) >> 5);
    const uint32_t beyond = S - wx < 8 ? (0xFFu << (S - wx)) & 0xFFu : 0u;
    uint32_t row[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool in = wy + i < S;
      const uint32_t lo = in ? q0[i * w] : 0xFFFFFFFFu, hi = in ? q1[i * w] : 0xFFFFFFFFu;
      row[i] = (__funnelshift_r(lo, hi, b & 31) & 0xFFu) | beyond;
    }
    win_lo = row[0] | row[1] << 8 | row[2] << 16 | row[3] << 24;
    win_hi = row[4] | row[5] << 8 | row[6] << 16 | row[7] << 24;
    // bit-plane maps: the maze's own door is open while its key is held
    const int dx = door_x - wx, dy = door_y - wy;
    if ((r.keys & 1) && (unsigned)dx < 8u && (unsigned)dy < 8u && p.step_bits && (unsigned)door_x < (unsigned)S &&
        (unsigned)door_y < (unsigned)S && map[door_y * S + door_x] == kDoor) {
      const int k = 8 * dy + dx;
      if (k < 32)
        win_lo &= ~(1u << k);
      else
        win_hi &= ~(1u << (k - 32));
    }
  };
  // solid3x3 of the lane's own cell; `reload`: the keys changed
  auto solid_around = [&](bool reload) {
    uint32_t m = 0u;
    const bool inner = (unsigned)(r.cx - 1) < (unsigned)(S - 2) && (unsigned)(r.cy - 1) < (unsigned)(S - 2);
    if (inner && (p.step_bits || r.keys == 0)) {
      if (reload || (unsigned)(r.cx - wx - 1) >= 6u || (unsigned)(r.cy - wy - 1) >= 6u) load_window();
      const int k = 8 * (r.cy - wy - 1) + r.cx - wx - 1;  // at most 45: the three rows end at bit 63
      const uint64_t v = (((uint64_t)win_hi << 32) | win_lo) >> k;
      const uint32_t u = (uint32_t)v;
      return (u & 7u) | ((u >> 8) & 7u) << 3 | ((u >> 16) & 7u) << 6;
    }
    wx = -64;  // the window is for the keys held then
    for (int k = 0; k < 9; ++k) {
      const int x = r.cx + k % 3 - 1, y = r.cy + k / 3 - 1;
      bool sld = true;  // outside the map
      if ((unsigned)x < (unsigned)S && (unsigned)y < (unsigned)S) {
        const int b = (y << sh) + x;
        sld = (plane[b >> 5] >> (b & 31)) & 1u;
        if (sld && r.keys != 0) {
          const int v = map[y * S + x];
          if (p.step_bits)  // the maze's own door
            sld = !((r.keys & 1) && x == door_x && y == door_y && v == kDoor);
          else  // byte maps: every locked door of a held colour is open
            sld = !(is_locked(v) && ((r.keys >> (v - kLocked)) & 1));
        }
      }
      m |= (sld ? 1u : 0u) << k;
    }
    return m;
  };
  uint32_t m = solid_around(true);
  const float rad = p.radius;
  const int horizon = p.horizon > 0 ? p.horizon : 0x7fffffff, tpr = p.tpr;
  auto turned = [&](int turn, int a) {
    turn += (a == 6 ? 1 : 0) - (a == 5 ? 1 : 0);
    return turn < 0 ? tpr - 1 : (turn == tpr ? 0 : turn);
  };
  bool fresh = true;  // the agent's cell has not been looked at for events in this launch
  bool go = on && stop > t_begin, bad = false;  // a stop lies in an earlier part, or at the first step of all
  const size_t first = (size_t)t_begin * stride + e, first_cam = (size_t)t_begin * p.n + e;
  float* rewards = p.rewards + first;
  uint8_t* dones = p.dones + first;
  uint4* cam_a = p.cam_a + first_cam;
  uint2* cam_b = p.cam_b + first_cam;
  int turn = turned(r.turn, (int)ahead[0]);
  float2 cs = __ldg(p.turn_cs + turn);
  for (int t0 = t_begin; t0 < t_end; t0 += kActAhead) {
#pragma unroll
    for (int i = 0; i < kActAhead; ++i) acts[32 * i + lane] = (uint8_t)ahead[i];
    act += kActAhead * stride;
#pragma unroll
    for (int i = 0; i < kActAhead; ++i) ahead[i] = t0 + kActAhead + i < t_end ? act[i * stride] : 0u;
    const int n = t_end - t0 < kActAhead ? t_end - t0 : kActAhead;
    if (!__any_sync(0xffffffffu, go)) break;
#pragma unroll 1
    for (int i = 0; i < n; ++i, rewards += stride, dones += stride, cam_a += p.n, cam_b += p.n) {
      const int a = acts[32 * i + lane];
      float c, s;
      heading_from(r, cs, c, s);
      const int turn_now = turn;
      turn = turned(turn, (int)(i + 1 < kActAhead ? acts[32 * (i + 1) + lane] : ahead[0]));
      cs = __ldg(p.turn_cs + turn);
      if (!go) continue;
      bad |= a > 6;
      Env q = r;
      const float2 d = move_delta(a, p.move, c, s);
      // x, then y: as try_move_x and try_move_y
      Env qx = r;
      qx.fx = __fadd_rn(r.fx, d.x);
      const bool free_x = !(rows3(m, span3(r.fy, rad)) & span3(qx.fx, rad));
      renormalise(qx.cx, qx.fx);
      q.fx = free_x ? qx.fx : r.fx;
      q.cx = free_x ? qx.cx : r.cx;
      Env qy = r;
      qy.fy = __fadd_rn(r.fy, d.y);
      // the columns under the box, as offsets from the start cell (its shifted span stays inside them)
      const bool free_y = !(rows3(m, span3(qy.fy, rad)) & ((span3(q.fx, rad) << (q.cx - r.cx + 1)) >> 1) & 7u);
      renormalise(qy.cy, qy.fy);
      q.fy = free_y ? qy.fy : r.fy;
      q.cy = free_y ? qy.cy : r.cy;
      const bool moved = q.cx != r.cx || q.cy != r.cy;
      uint32_t picked = 0u;
      bool goal = false;
      if (moved || fresh) {  // events happen where an agent enters a cell
        const int here = q.cx | q.cy << 8;
        for (int k = 0; k < n_ev; ++k) {
          const int v = (int)spr[32 * k + lane];
          if ((v & 0xffff) != here) continue;
          const int kc = key_colour(v >> 16);
          if (kc >= 0 && !((q.keys >> kc) & 1)) picked |= 1u << kc;
          goal = goal || kc < 0;
        }
        fresh = false;
      }
      q.t += 1;
      if (goal || q.t >= horizon) {  // left to the env kernel, from before this step
        stop = t0 + i;
        go = false;
        continue;
      }
      q.keys |= (int)picked;
      q.turn = turn_now;
      r = q;
      if (moved || picked) m = solid_around(picked != 0u);
      *rewards = p.reward_lut[picked ? 1 : 0];
      *dones = 0;
      *cam_a = make_uint4((uint32_t)r.cx | (uint32_t)r.cy << 16, __float_as_uint(r.fx), __float_as_uint(r.fy),
                          __float_as_uint(c));
      *cam_b = make_uint2(__float_as_uint(s), (uint32_t)r.keys | (uint32_t)(r.t & 3) << 8);
    }
  }
  if (bad) atomicOr(p.err, 1u);  // an action outside 0..6 was taken as a no-op
  if (on) {
    const State& st = p.st;
    st.cell_x[e] = (int16_t)r.cx;
    st.cell_y[e] = (int16_t)r.cy;
    st.frac_x[e] = r.fx;
    st.frac_y[e] = r.fy;
    st.turn[e] = (int16_t)r.turn;
    st.t[e] = r.t;
    st.flags[e] = (uint8_t)r.keys;
    p.stop[e] = stop;
  }
  const uint32_t left = __ballot_sync(0xffffffffu, on && stop < p.steps);
  if (lane == 0 && on) p.ended[e >> 5] = left;  // lane 0's env is a multiple of 32
}

// Frames of steps t0 .. t1 - 1 of env e from their camera records, in a part
// that ends at t_part. The walk of the next part may be storing a new stop
// step meanwhile: the old and the new one both lie at or beyond t_part then.
template <int GRAY>
__device__ __forceinline__ void draw_env(const Params& p, int e, int t0, int t1, int t_part, uint8_t* wbase,
                                         int lane) {
  int stop = *reinterpret_cast<volatile int32_t*>(p.stop + e);
  if (stop > t_part) stop = t_part;
  if (t1 > stop) t1 = stop;
  if (t0 >= t1) return;
  const WarpSmem ws{wbase, fill_lane(p, lane)};
  const size_t frame_bytes = (size_t)3 * p.H * p.W;
  const uint4* cam_a = p.cam_a + e;
  const uint2* cam_b = p.cam_b + e;
  uint4 a = __ldcg(cam_a + (size_t)t0 * p.n);
  uint2 b = __ldcg(cam_b + (size_t)t0 * p.n);
  const float2 k01 = col_k_pair(p, lane);
  {
    Prefetch q;  // map, objects and sprites only
    q.obj = lane < 6 ? (int)p.st.obj[6 * (size_t)e + lane] : (lane == 6 ? (int)p.st.nspr[e] : 0);
    q.spr = make_float4(0.f, 0.f, 0.f, 0.f);
    if (lane < p.K) {
      const size_t i = (size_t)e * p.K + lane;
      q.spr = make_float4(p.st.spr_x[i], p.st.spr_y[i], (float)p.st.spr_type[i], 0.f);
    }
    q.m0 = q.m1 = make_uint4(0u, 0u, 0u, 0u);
    if (small_map<MAP_BITS>(p) && lane < p.plane_words) q.m0.x = plane_of(p, e)[lane];
    stage_prefetched<MAP_BITS>(p, ws, e, q, lane);  // ends with __syncwarp
  }
  int keys = 0, slot = 0;
  for (int t = t0; t < t1; ++t) {
    Env r;
    r.cx = (int)(a.x & 0xffffu);
    r.cy = (int)(a.x >> 16);
    r.fx = __uint_as_float(a.y);
    r.fy = __uint_as_float(a.z);
    const float c = __uint_as_float(a.w), s = __uint_as_float(b.x);
    r.keys = (int)(b.y & 7u);
    r.t = 4 + (int)(b.y >> 8);  // only its plane matters: an episode's first frame is never drawn here
    if (t + 1 < t1) {
      a = __ldcg(cam_a + (size_t)(t + 1) * p.n);
      b = __ldcg(cam_b + (size_t)(t + 1) * p.n);
    }
    if (__builtin_expect(r.keys != keys, 0)) {
      keys = r.keys;
      open_doors<MAP_BITS>(p, e, keys, ws, lane);
      mark_border<MAP_BITS>(p, ws, lane);
    }
    render_env<MODE_ROLLOUT, MAP_BITS, 1, GRAY>(p, e, r, c, s, ws, lane, slot,
                                                p.frames + (size_t)t * p.frame_step + (size_t)e * frame_bytes, k01,
                                                t + 4 >= stop);
    __syncwarp();
  }
  // shared memory stays allocated until the bulk stores have read it
  if (lane == 0) bulk_wait_read_all();
}

// Steps of draw chunk k of a part (see DrawPart).
__device__ __forceinline__ void chunk_steps(const DrawPart& d, int k, int& t0, int& t1) {
  int n = d.chunk;
  t0 = d.t0 + k * d.chunk;
  if (k >= d.n_chunks) {
    t0 = d.t0 + d.n_chunks * d.chunk + 2 * (k - d.n_chunks);
    n = 2;
    if (k >= d.n_chunks + d.n_pairs) {
      t0 = d.t0 + d.n_chunks * d.chunk + 2 * d.n_pairs + (k - d.n_chunks - d.n_pairs);
      n = 1;
    }
  }
  t1 = t0 + n < d.t1 ? t0 + n : d.t1;
}
__host__ __device__ __forceinline__ int chunk_count(const DrawPart& d) {
  const int singles = d.t1 - d.t0 - d.n_chunks * d.chunk - 2 * d.n_pairs;
  return d.n_chunks + d.n_pairs + (singles > 0 ? singles : 0);
}

// Every kernel here is a programmatic dependent: its blocks may be resident
// while the kernel before it drains, and wait until that one has completed and
// its writes are visible. They release their own dependents only then, so no
// kernel starts before all but the one ahead of it have completed.
__device__ __forceinline__ void wait_and_release() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// One launch: blocks of two warps. The first part.walk_blocks of them walk
// steps walk_t0 .. walk_t1 - 1 of 64 envs each; the others draw, each warp one
// (env, chunk): chunk by chunk, so that the shortest chunks come last.
template <int GRAY>
__global__ void __launch_bounds__(kThreads, kMinBlocksPerSm / kWarpsPerBlock)
    rollout_kernel(const __grid_constant__ Params p, const __grid_constant__ DrawPart part) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint8_t* const wbase = smem_raw + warp * p.warp_bytes;
  if ((int)blockIdx.x < part.walk_blocks) {
    wait_and_release();
    const int e = ((int)blockIdx.x * kWarpsPerBlock + warp) * 32 + lane;
    walk_envs<GRAY>(p, e, part.walk_t0, part.walk_t1, reinterpret_cast<uint32_t*>(wbase), lane);
    return;
  }
  write_palette(p, WarpSmem{wbase, FillLane{}}, lane);
  wait_and_release();
  const int b = (int)blockIdx.x - part.walk_blocks;
  const int pairs = (p.n + kWarpsPerBlock - 1) / kWarpsPerBlock;
  const int chunk = b / pairs, e = (b - chunk * pairs) * kWarpsPerBlock + warp;
  int t0, t1;
  chunk_steps(part, chunk, t0, t1);
  if (e < p.n) draw_env<GRAY>(p, e, t0, t1, part.t1, wbase, lane);
}

// The same over the groups of a batch: the walk blocks of every group first,
// then the draw blocks, the groups with the largest frames first.
template <int GRAY>
__global__ void __launch_bounds__(kThreads, kMinBlocksPerSm / kWarpsPerBlock)
    batch_rollout_kernel(const __grid_constant__ BatchParams bp, const __grid_constant__ BatchDrawPart parts) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint8_t* const wbase = smem_raw + warp * bp.warp_bytes;
  int g = 0;
  if ((int)blockIdx.x < parts.walk_blocks) {
    while (g + 1 < bp.n_groups && (int)blockIdx.x >= parts.first_walk[g + 1]) ++g;
    wait_and_release();
    const int e = (((int)blockIdx.x - parts.first_walk[g]) * kWarpsPerBlock + warp) * 32 + lane;
    walk_envs<GRAY>(bp.g[g], e, parts.g[g].walk_t0, parts.g[g].walk_t1, reinterpret_cast<uint32_t*>(wbase), lane);
    return;
  }
  while (g + 1 < bp.n_groups && (int)blockIdx.x >= parts.first_draw[g + 1]) ++g;
  const Params& p = bp.g[g];
  write_palette(p, WarpSmem{wbase, FillLane{}}, lane);
  wait_and_release();
  const int b = (int)blockIdx.x - parts.first_draw[g];
  const int pairs = (p.n + kWarpsPerBlock - 1) / kWarpsPerBlock;
  const int chunk = b / pairs, e = (b - chunk * pairs) * kWarpsPerBlock + warp;
  int t0, t1;
  chunk_steps(parts.g[g], chunk, t0, t1);
  if (e < p.n) draw_env<GRAY>(p, e, t0, t1, parts.g[g].t1, wbase, lane);
}

template <class... P>
cudaError_t launch_dependent(void (*kernel)(P...), int grid, int smem, cudaStream_t stream, const P&... params) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, params...);
}

constexpr int kEnvsPerWalkBlock = 32 * kWarpsPerBlock;

// Large chunks stage a map and its sprites once for many frames; small ones
// leave less running at the end of the launch, and fill the chip when there
// are few envs.
void choose_chunks(DrawPart& d, int n, int slots) {
  const int steps = d.t1 - d.t0;
  const int64_t frames = (int64_t)n * steps;
  int c = (int)(frames / ((int64_t)slots * 6));
  c = c < 1 ? 1 : (c > 4 ? 4 : c);
  // about one frame per slot in single steps at the end, as many in pairs before
  int singles = c == 1 ? steps : (slots + n - 1) / n;
  int pairs = c <= 2 ? 0 : singles;
  if (singles > steps) singles = steps;
  if (singles + 2 * pairs > steps) pairs = (steps - singles) / 2;
  const int big = (steps - singles - 2 * pairs) / c;
  if (c > 2) pairs = (steps - big * c - singles) / 2;  // what is left over goes in pairs and a single step
  d.chunk = c;
  d.n_chunks = big;
  d.n_pairs = pairs;
}

// The parts of a rollout of `steps` steps that writes frame_bytes a step, in
// frames of at most frame_px pixels: each part's walk takes as long as the part
// before takes to draw, so that only the first part's walk is waited for. A
// step of the walk takes about 1.2 us, frames go out at about 7 TB/s. Every
// part's end costs a part of the time its last frames take on their warps
// (about 3 us for 64 x 64): the rollout stays whole where that is not well
// below the walk, and where the draw is the shorter of the two. (4096 envs, 64
// x 64: 20 steps take 168 us whole, 160 in parts of 3 and 17; 16,384 envs,
// 128 x 128, 8 steps, building next episodes: 1.41 ms whole, 1.49
// in parts of 2 and 6.) Writes the parts' ends to `ends` and returns
// their number.
int choose_parts(int steps, int64_t frame_bytes, int frame_px, int* ends) {
  const double walk_us = 1.2, ratio = (double)frame_bytes / 7.0e6 / walk_us;  // draw over walk of a step
  const double end_us = 3.0 * frame_px / 4096;
  int n = 0;
  if (ratio >= 2.0 && walk_us * steps > 4.0 * end_us) {
    double reach = 1.0;  // steps that parts of a one-step first part would cover
    double last = 1.0;
    int parts = 1;
    for (; parts < kMaxParts - 1 && reach * 3.0 < steps; ++parts) {
      last *= ratio;
      reach += last;
    }
    int at = 0;
    for (double len = steps / reach; n < parts - 1; ++n, len *= ratio) {
      at += (int)(len + 0.99);
      if (at >= steps) break;
      ends[n] = at;
    }
  }
  ends[n++] = steps;
  return n;
}
}  // namespace

// Two passes take two launches more and the walk's chain, some 6 us a call, and
// save per step what a warp's frame takes beyond its share of a full chip. So
// the line lies higher where frames are small, in mazes, whose rays are short,
// and where a step's warps just fill the chip (one round, none waiting), which
// suits the env kernel best. Calls back to back, us, env kernel / two passes:
//   mazes of side 32, 32 x 32: 600 envs 3 steps 11.9 / 12.3, 4 14.1 / 13.1;
//     4096 envs 4 steps 22.9 / 27.8, 8 40.9 / 44.6, 10 51.5 / 52.8; 64 x 64: 1200
//     envs 2 steps 13.4 / 15.0, 3 19.3 / 17.4; 4096 envs 3 steps 30.3 / 34.0, 6
//     55.9 / 55.6; 128 x 128: 2400 envs 2 steps 43.4 / 54.9, 4 81.3 / 82.1; 4096
//     envs 2 steps 70.1 / 71.7, 3 102.4 / 98.1
//   rooms of side 64 with sprites, 32 x 32: 1200 envs 2 steps 12.0 / 13.1, 3
//     16.3 / 14.1; 64 x 64: 4096 envs 3 steps 35.8 / 38.9, 5 56.2 / 56.2
// In mazes of four nodes an episode lasts a few dozen steps, so most envs leave
// the walk, and their rest runs as in the env kernel alone: 64 x 64, 4096 envs
// 8 steps 80 / 101, 20 steps 194 / 223, 48 454 / 478; 600 envs 8 steps 47 / 41.
int rollout_min_steps(int task, int side, int n, int px, int slots) {
  const bool small = px <= 32 * 32, maze = task != 0;
  const bool fits = n <= slots, fills = fits && n > slots * 3 / 10;
  if (maze && side < 8) {
    if (px > 64 * 64) return fits && n > slots * 2 / 5 ? 32 : 2;
    return !fits ? 16 : (n > slots / 4 ? 48 : (small ? 12 : 4));
  }
  if (px > 64 * 64) return fits && n > slots * 2 / 5 ? 3 : 2;
  if (!fits) return small ? (maze ? 6 : 4) : 3;
  const int few = (small ? 3 : 2) + (maze ? 1 : 0);
  if (!fills) return few;
  const int at = maze ? 2 : (small ? 3 : 1), slope = maze && small ? 9 : 4;  // from few envs to a full chip
  const int line = at + (int)((int64_t)slope * n / slots);
  return line > few ? line : few;
}

int rollout_segment(int n) {
  // 64 MB of camera records, but at least 16 steps (more than that above 174,762 envs: 384 bytes an env)
  const int64_t fit = ((int64_t)64 << 20) / (24 * (int64_t)n);
  return fit > 128 ? 128 : (fit < 16 ? 16 : (int)fit);
}

bool rollout_wanted(int task) { return task != kTaskAscii; }  // maps that open doors change between frames

size_t rollout_bytes(int n) {
  const size_t N = (size_t)n, R = (size_t)rollout_segment(n);
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  return up(16 * N * R) + up(8 * N * R) + up(4 * N) + up(4 * ((N + 31) / 32));
}

void rollout_place(Params& p, uint8_t* mem) {
  const size_t N = (size_t)p.n, R = (size_t)rollout_segment(p.n);
  auto take = [&](size_t bytes) {
    uint8_t* at = mem;
    mem += (bytes + 255) & ~(size_t)255;
    return at;
  };
  p.cam_a = reinterpret_cast<uint4*>(take(16 * N * R));
  p.cam_b = reinterpret_cast<uint2*>(take(8 * N * R));
  p.stop = reinterpret_cast<int32_t*>(take(4 * N));
  p.ended = reinterpret_cast<uint32_t*>(take(4 * ((N + 31) / 32)));
}

void rollout_layout(Params& q, size_t smem_per_sm, size_t reserved) {
  q.step_bits = q.map_bits;
  q.map_bits = 1;  // the draw holds every map as a bit plane
  host::choose_rows(q, 32, kWarpsPerBlock, kMinBlocksPerSm, smem_per_sm, reserved);
  if (q.warp_bytes < walk_warp_bytes(q.K)) q.warp_bytes = walk_warp_bytes(q.K);
}

cudaError_t rollout_prepare(const Params& q) {
  return raise_smem_limit(q.gray ? rollout_kernel<1> : rollout_kernel<0>);
}

RolloutParts rollout_parts(const Params& q) {
  RolloutParts parts;
  parts.n = choose_parts(q.steps, (int64_t)q.n * 3 * q.H * q.W, q.H * q.W, parts.ends);
  return parts;
}

cudaError_t rollout_launch(const Params& q, const RolloutParts& parts, int i, int slots, cudaStream_t stream) {
  DrawPart d = {};
  d.walk_blocks = i < parts.n ? (q.n + kEnvsPerWalkBlock - 1) / kEnvsPerWalkBlock : 0;
  d.walk_t0 = i > 0 ? parts.ends[i - 1] : 0;
  d.walk_t1 = i < parts.n ? parts.ends[i] : 0;
  d.t0 = i > 1 ? parts.ends[i - 2] : 0;
  d.t1 = i > 0 ? parts.ends[i - 1] : 0;
  choose_chunks(d, q.n, slots);
  const int64_t grid = d.walk_blocks + (int64_t)((q.n + kWarpsPerBlock - 1) / kWarpsPerBlock) * chunk_count(d);
  return launch_dependent(q.gray ? rollout_kernel<1> : rollout_kernel<0>, (int)grid, block_smem_bytes(q), stream, q, d);
}

cudaError_t batch_rollout_prepare(const BatchParams& bq) {
  bool gray = false;
  for (int g = 0; g < bq.n_groups; ++g) gray = gray || bq.g[g].gray;
  return raise_smem_limit(gray ? batch_rollout_kernel<2> : batch_rollout_kernel<0>);
}

cudaError_t batch_rollout_launch(const BatchParams& bq, int steps, int slots, cudaStream_t stream, int* launches) {
  bool gray = false;
  int64_t frame_bytes = 0;
  int frame_px = 0;
  for (int g = 0; g < bq.n_groups; ++g) {
    gray = gray || bq.g[g].gray;
    if (!bq.g[g].stop) continue;
    const int px = bq.g[g].H * bq.g[g].W;
    frame_bytes += (int64_t)bq.g[g].n * 3 * px;
    frame_px = px > frame_px ? px : frame_px;
  }
  if (frame_bytes == 0) return cudaSuccess;  // the batched kernel runs every group alone
  int ends[kMaxParts];
  const int parts = choose_parts(steps, frame_bytes, frame_px, ends);
  for (int i = 0; i <= parts; ++i) {
    BatchDrawPart d = {};
    int64_t blocks = 0;
    for (int g = 0; g < bq.n_groups; ++g) {
      d.first_walk[g] = (int32_t)blocks;
      d.g[g].walk_t0 = i > 0 ? ends[i - 1] : 0;
      d.g[g].walk_t1 = i < parts ? ends[i] : 0;
      if (i < parts && bq.g[g].stop) blocks += (bq.g[g].n + kEnvsPerWalkBlock - 1) / kEnvsPerWalkBlock;
    }
    d.walk_blocks = (int32_t)blocks;
    for (int g = 0; g < bq.n_groups; ++g) {
      const Params& q = bq.g[g];
      d.first_draw[g] = (int32_t)blocks;
      d.g[g].t0 = i > 1 ? ends[i - 2] : 0;
      d.g[g].t1 = i > 0 ? ends[i - 1] : 0;
      // only the last groups' chunks end the launch
      choose_chunks(d.g[g], q.n, g + 1 < bq.n_groups ? 1 + slots / bq.n_groups : slots);
      if (q.stop) blocks += (int64_t)((q.n + kWarpsPerBlock - 1) / kWarpsPerBlock) * chunk_count(d.g[g]);
    }
    cudaError_t err = launch_dependent(gray ? batch_rollout_kernel<2> : batch_rollout_kernel<0>, (int)blocks,
                                       bq.warp_bytes * kWarpsPerBlock, stream, bq, d);
    if (err != cudaSuccess) return err;
    ++*launches;
  }
  return cudaSuccess;
}
}  // namespace jx
